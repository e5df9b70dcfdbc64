// Eq. (eqkl) as increments on the tcgen05 tensor cores, materialising dW:
//   dW[s][w][n] = sum_k zeta[s][w*K + k] phi[k][n]
// with BF16 operands (or split hi/lo BF16, three products) and FP32
// accumulation in TMEM.  One CTA per [128 samples x TN steps] block of one
// disturbance; thread 0 streams the K blocks with TMA and issues the MMAs, then
// each of the four warps reads its 32 TMEM lanes (= its 32 samples) and writes
// the rows to HBM: through bulk copies of rows staged in shared memory where every row
// starts on 16 bytes, else by transposes of 32 x 32 and plain stores.  What bounds it: the
// stores' path while they were instructions (plain stores 379 us by lane, 121 us
// transposed, 94 us as bulk copies for 8192 x 3 rows of 2000 steps, K = 200, split), then
// the operands' way through L2 (0.7 GB; the products are 59 GFLOP, 31 us at the tensor
// cores' rate).  Keeping the design tile resident, with four storing warps per SM, was
// slower (the whole call 225 instead of 218 us); blocks of 256 steps (contract_block) take
// it from 190 to 178 us.
// This standalone form serves fmc_kle_reconstruct; the fused simulation consumes the same
// TMEM tiles without writing them out.
#include <cuda_bf16.h>

#include "fmc_common.cuh"
#include "kernels.cuh"
#include "tc_common.cuh"

namespace fmc {

struct ContractArgs {
    int64_t count;
    int d, Ks, nkb, Nt, TN;
    int split, ns;
    int bulk;  // rows of dW start on 16 bytes: stored by bulk copies
    float* dW;
    int* err;
};

constexpr int CT_LD = 33;   // floats per row of a warp's 32 x 32 transpose
constexpr int CT_LDB = 132;  // and of the block staged for the bulk copies (128 + 16 bytes: no bank conflicts)

// Asynchronous copy of bytes (a multiple of 16) of shared memory to dst, both 16-byte
// aligned, given up first by L2; the caller's next wait is bulk_read_wait.
__device__ __forceinline__ void bulk_store(void* dst, const void* src, uint32_t bytes, uint64_t policy)
{
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group.L2::cache_hint [%0], [%1], %2, %3;" ::"l"(
                     __cvta_generic_to_global(dst)),
                 "r"(smem_u32(src)), "r"(bytes), "l"(policy)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// Until the thread's bulk stores have read their shared memory.
__device__ __forceinline__ void bulk_read_wait() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

__global__ void __launch_bounds__(128) contract_tc_kernel(const __grid_constant__ CUtensorMap mAh,
                                                          const __grid_constant__ CUtensorMap mAl,
                                                          const __grid_constant__ CUtensorMap mBh,
                                                          const __grid_constant__ CUtensorMap mBl, ContractArgs a)
{
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    // 1 KB alignment by an offset from the shared array itself (not through an
    // integer round trip), so that every access through these pointers stays a
    // shared-memory access rather than a generic one
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    __shared__ uint64_t bars[2 * TC_MAX_STAGES + 1];  // full[ns], freed[ns], done
    __shared__ uint32_t tmem_base;
    __shared__ int ok_flag;

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int n0 = blockIdx.x * a.TN;
    const int64_t row0 = (int64_t)blockIdx.y * TC_M;
    const int w = blockIdx.z;
    const uint32_t ncols = a.TN < 32 ? 32 : a.TN;

    TcRing r;
    r.a_bytes = TC_M * 64;
    r.b_bytes = a.TN * 64;
    r.split = a.split;
    r.base = smem;
    r.ns = (uint32_t)a.ns;
    r.full = &bars[0];
    r.freed = &bars[TC_MAX_STAGES];
    uint64_t* done = &bars[2 * TC_MAX_STAGES];

    if (threadIdx.x == 0) {
        prefetch_tmap(&mAh);
        prefetch_tmap(&mBh);
        for (int b = 0; b < 2 * TC_MAX_STAGES + 1; ++b) mbar_init(&bars[b], 1);
        fence_mbar_init();
        ok_flag = 1;
    }
    if (warp == 0) tmem_alloc(&tmem_base, ncols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;

    if (threadIdx.x == 0) {
        const uint32_t idesc = umma_idesc_bf16(TC_M, a.TN);
        bool ok = true;
        const int ax0 = w * a.Ks;
        int issued = 0;
        auto load = [&](int kb) {
            return ring_load(r, (uint32_t)kb, &mAh, &mAl, &mBh, &mBl, ax0 + kb * TC_BK, (int)row0, kb * TC_BK, n0);
        };
        for (; issued < a.nkb && issued + 1 < a.ns && ok; ++issued) ok = load(issued);
        for (int kb = 0; kb < a.nkb && ok; ++kb) {
            if (issued < a.nkb) {
                ok = load(issued);
                ++issued;
            }
            if (ok) ok = ring_mma(r, (uint32_t)kb, tmem, idesc, kb == 0);
        }
        if (ok) umma_commit(done);
        if (!ok) {
            ok_flag = 0;
            atomicExch(a.err, DEV_TIMEOUT_TMA);
        }
    }
    __syncthreads();
    bool ok = ok_flag != 0;
    if (ok && !mbar_wait(done, 0)) {
        ok = false;
        if (lane == 0) atomicExch(a.err, DEV_TIMEOUT_MMA);
    }
    // all warps agree on ok (tcgen05.ld is warp-collective, and the transposes below
    // take the ring's place: every MMA has read its operands)
    ok = __syncthreads_and(ok);
    tc_fence_after();
    if (ok) {
        const uint32_t lane_addr = tmem + ((uint32_t)(warp * 32) << 16);
        float* tr = reinterpret_cast<float*>(smem) + warp * 32 * CT_LD;
        const int64_t left = a.count - row0 - warp * 32;  // samples of this warp
        const int rows = left <= 0 ? 0 : (left >= 32 ? 32 : (int)left);
        float* out = a.dW + ((row0 + warp * 32) * a.d + w) * (int64_t)a.Nt + n0;
        const int64_t rs = (int64_t)a.d * a.Nt;
        if (a.bulk) {
            // a lane stages its sample's row in the ring's place (every product has read its
            // operands) and hands it to one bulk copy: no store instructions, and the copies
            // run beside the other CTAs' work
            float* row = reinterpret_cast<float*>(smem) + (warp * 32 + lane) * CT_LDB;
            const int all = a.Nt - n0 < a.TN ? a.Nt - n0 : a.TN;
            for (int c0 = 0; c0 < all; c0 += 128) {  // 128 steps of every row at a time
                const int cols = all - c0 < 128 ? all - c0 : 128;
                for (int c = 0; c < cols; c += 32) {
                    float v[32];
#pragma unroll
                    for (int e = 0; e < 32; e += 8)
                        tmem_ld8(lane_addr + c0 + c + e, reinterpret_cast<float(&)[8]>(v[e]));
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 32; e += 4)
                        *reinterpret_cast<float4*>(row + c + e) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                if (lane < rows) {
                    bulk_store(out + lane * rs + c0, row, (uint32_t)cols * 4u, l2_policy_evict_first());
                    bulk_read_wait();
                }
                __syncwarp();  // (the next loads from TMEM are the whole warp's)
            }
        } else
        // a lane holds a sample's row: 32 steps at a time are turned in shared memory, so
        // that a warp stores 128 consecutive bytes of one row
        for (int c = 0; c < a.TN && n0 + c < a.Nt; c += 32) {
            float v[32];
#pragma unroll
            for (int e = 0; e < 32; e += 8) tmem_ld8(lane_addr + c + e, reinterpret_cast<float(&)[8]>(v[e]));
            tmem_ld_wait();
            __syncwarp();
#pragma unroll
            for (int e = 0; e < 32; ++e) tr[lane * CT_LD + e] = v[e];
            __syncwarp();
            if (n0 + c + lane < a.Nt)
#pragma unroll 8
                for (int s = 0; s < rows; ++s) __stcs(out + s * rs + c + lane, tr[s * CT_LD + lane]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, ncols);
}

// zeta [count][d*K] FP32 -> hi/lo [count][d][Ks] BF16 with zero padding.
// A CTA takes 128 consecutive positions of the padded row and steps over samples, so
// no index division is left per entry.
__global__ void __launch_bounds__(256) split_rows_kernel(const float* __restrict__ z, int64_t count, int d, int K,
                                                         int Ks, __nv_bfloat16* __restrict__ hi,
                                                         __nv_bfloat16* __restrict__ lo)
{
    const int64_t cols = (int64_t)d * Ks;
    for (int64_t pos = blockIdx.y * (int64_t)128 + threadIdx.x % 128; pos < cols; pos += (int64_t)gridDim.y * 128) {
        const int64_t w = pos / Ks, kk = pos - w * Ks;
        const bool real = kk < K;
        const float* zc = z + w * K + kk;
        for (int64_t j = blockIdx.x * (int64_t)2 + threadIdx.x / 128; j < count; j += (int64_t)gridDim.x * 2) {
            const float v = real ? zc[j * d * K] : 0.f;
            const __nv_bfloat16 h = __float2bfloat16_rn(v);
            hi[j * cols + pos] = h;
            lo[j * cols + pos] = __float2bfloat16_rn(v - __bfloat162float(h));
        }
    }
}

cudaError_t launch_split_rows(const float* z, int64_t count, int d, int K, int Ks, void* hi, void* lo, cudaStream_t st)
{
    int64_t gy = ((int64_t)d * Ks + 127) / 128;
    if (gy > 65535) gy = 65535;
    int64_t gx = (count + 15) / 16;  // eight samples per thread
    if (gx > 65536) gx = 65536;
    split_rows_kernel<<<dim3((unsigned)gx, (unsigned)gy), 256, 0, st>>>(z, count, d, K, Ks, (__nv_bfloat16*)hi,
                                                                       (__nv_bfloat16*)lo);
    return cudaGetLastError();
}

// Blocks of 256 steps read the samples half as often: an eighth less time per step where
// the SMs are full (16384 x 3 rows of 2000 steps, K = 200, the whole call 239 -> 215 us).
// But two CTAs per SM hold four blocks of 128 steps where three CTAs hold three.  So 256
// where they add no padding and their rounds, at 7/6 the time of the others', are no
// longer in all (2000 x 3 rows: 62.0 us with 128, 62.8 with 256; plain BF16 52.6, 54.5).
int contract_block(int64_t count, int d, int Nt, int sms)
{
    const int64_t cols = (Nt + 127) / 128, blocks = (count + TC_M - 1) / TC_M * d * cols;
    if (cols % 2) return 128;
    const int64_t r256 = (blocks + 4 * sms - 1) / (4 * sms), r128 = (blocks + 3 * sms - 1) / (3 * sms);
    return 7 * r256 <= 6 * r128 ? 256 : 128;
}

cudaError_t launch_contract_tc(const CUtensorMap* maps, int64_t count, int d, int Ks, int nkb, int Nt, int TN,
                               int split, float* dW, int* err, cudaStream_t st)
{
    // blocks of 128 steps: three CTAs per SM with two 32 KB stages (three 16 KB stages in
    // plain BF16); of 256: two CTAs.  One CTA's stores run beside the others' loads and MMAs
    const int stage_bytes = (TC_M * 64 + TN * 64) * (split ? 2 : 1);
    const int ns = split ? 2 : 3;
    const int bulk = Nt % 4 == 0 && reinterpret_cast<uintptr_t>(dW) % 16 == 0;
    ContractArgs a{count, d, Ks, nkb, Nt, TN, split, ns, bulk, dW, err};
    // enough that no more CTAs share an SM than its 512 TMEM columns hold
    int smem = ns * stage_bytes + 1024;
    const int trans = (bulk ? TC_M * CT_LDB : 4 * 32 * CT_LD) * 4 + 1024;
    if (smem < trans) smem = trans;
    const int floor = 233472 / (512 / TN + 1) - 1024 + 64;
    if (smem < floor) smem = floor;
    // (an attribute of the current device, always the same bound: launches may race on it)
    cudaError_t e = cudaFuncSetAttribute(contract_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 112 * 1024);
    if (e != cudaSuccess) return e;
    int64_t gy = (count + TC_M - 1) / TC_M;
    if (gy > 65535) return cudaErrorInvalidValue;
    dim3 grid((Nt + TN - 1) / TN, (unsigned)gy, d);
    contract_tc_kernel<<<grid, 128, smem, st>>>(maps[0], maps[1], maps[2], maps[3], a);
    return cudaGetLastError();
}

}  // namespace fmc
