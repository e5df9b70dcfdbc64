// Eq. (eqkl) as increments, plain FP32 form: dW = Z . Phi with Z the
// coefficients viewed as [count*d][K] and Phi the increment basis [K][Nt];
// dW [count*d][Nt]; and R Q^-T of the correlation-reducing permutation.
#include "fmc_common.cuh"
#include "kernels.cuh"

namespace fmc {

// A register-tiled SIMT GEMM, bound by the FP32 FMA pipe: 128 x 128 outputs per CTA of
// 256 threads, 8 x 8 per thread, so that a K step is 64 FMA per four 16-byte
// shared loads.  K goes through two shared buffers 16 at a time, the next block's
// global loads in flight (registers) while this one is multiplied: one barrier per
// block.  Every output sums its products one by one in the order of k, so neither the
// tile nor the K blocks show in the result.  Rows of A and B, whose lengths need not
// be multiples of four, are read 16 bytes at a time where VEC (all row starts are
// 16-byte aligned).  UPPER (B upper triangular): a column tile stops at its last
// non-zero row.
// Measured (GB300): 16384 x 600 x 600 upper triangular 243 us.
constexpr int SG_BM = 128, SG_BN = 128, SG_BK = 16, SG_LD = SG_BM + 4;

template <bool VEC, bool UPPER>
__global__ void __launch_bounds__(256, 2) sgemm_nn_kernel(int64_t R, int Ncols, int K, const float* __restrict__ A,
                                                          const float* __restrict__ B, float* __restrict__ C)
{
    __shared__ __align__(16) float As[2][SG_BK][SG_LD];  // [k][row]
    __shared__ __align__(16) float Bs[2][SG_BK][SG_BN];
    const int tid = threadIdx.x;
    const int tx = tid % 16, ty = tid / 16;
    const int64_t row0 = (int64_t)blockIdx.y * SG_BM;
    const int col0 = blockIdx.x * SG_BN;
    const int kend = UPPER && col0 + SG_BN < K ? col0 + SG_BN : K;
    // this thread's share of a block: 8 values of A's row ar from k = ak, 8 of B's row bk from column bc
    const int ar = tid / 2, ak = (tid % 2) * 8;
    const int bk = tid / 16, bc = (tid % 16) * 8;
    const bool arow = row0 + ar < R;
    const float* ap = A + (row0 + ar) * (int64_t)K + ak;
    const float* bp = B + (int64_t)bk * Ncols + col0 + bc;
    float av[8], bv[8];
    auto load = [&](int k0) {
        if (VEC) {
            // (K and Ncols are multiples of four: a group of four is inside or outside)
#pragma unroll
            for (int e = 0; e < 8; e += 4) {
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f), u = v;
                if (arow && k0 + ak + e < kend) v = *reinterpret_cast<const float4*>(ap + k0 + e);
                if (k0 + bk < kend && col0 + bc + e < Ncols)
                    u = *reinterpret_cast<const float4*>(bp + (int64_t)k0 * Ncols + e);
                av[e] = v.x, av[e + 1] = v.y, av[e + 2] = v.z, av[e + 3] = v.w;
                bv[e] = u.x, bv[e + 1] = u.y, bv[e + 2] = u.z, bv[e + 3] = u.w;
            }
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                av[e] = arow && k0 + ak + e < kend ? ap[k0 + e] : 0.f;
                bv[e] = k0 + bk < kend && col0 + bc + e < Ncols ? bp[(int64_t)k0 * Ncols + e] : 0.f;
            }
        }
    };
    auto store = [&](int b) {
#pragma unroll
        for (int e = 0; e < 8; ++e) As[b][ak + e][ar] = av[e];
        *reinterpret_cast<float4*>(&Bs[b][bk][bc]) = make_float4(bv[0], bv[1], bv[2], bv[3]);
        *reinterpret_cast<float4*>(&Bs[b][bk][bc + 4]) = make_float4(bv[4], bv[5], bv[6], bv[7]);
    };
    float acc[8][8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;

    load(0);
    store(0);
    __syncthreads();
    int buf = 0;
    for (int k0 = 0; k0 < kend; k0 += SG_BK, buf ^= 1) {
        const bool more = k0 + SG_BK < kend;
        if (more) load(k0 + SG_BK);
#pragma unroll
        for (int kk = 0; kk < SG_BK; ++kk) {
            float a[8], b[8];
            *reinterpret_cast<float4*>(a) = *reinterpret_cast<const float4*>(&As[buf][kk][ty * 4]);
            *reinterpret_cast<float4*>(a + 4) = *reinterpret_cast<const float4*>(&As[buf][kk][64 + ty * 4]);
            *reinterpret_cast<float4*>(b) = *reinterpret_cast<const float4*>(&Bs[buf][kk][tx * 4]);
            *reinterpret_cast<float4*>(b + 4) = *reinterpret_cast<const float4*>(&Bs[buf][kk][64 + tx * 4]);
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        if (more) store(buf ^ 1);
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int64_t gr = row0 + ((i < 4) ? ty * 4 + i : 64 + ty * 4 + (i - 4));
        if (gr >= R) continue;
#pragma unroll
        for (int jh = 0; jh < 8; jh += 4) {
            const int gc = col0 + (jh ? 64 : 0) + tx * 4;
            float* o = C + gr * Ncols + gc;
            if (VEC) {
                if (gc < Ncols)
                    *reinterpret_cast<float4*>(o) =
                        make_float4(acc[i][jh], acc[i][jh + 1], acc[i][jh + 2], acc[i][jh + 3]);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (gc + j < Ncols) o[j] = acc[i][jh + j];
            }
        }
    }
}

cudaError_t launch_sgemm_nn(int64_t R, int Ncols, int K, const float* A, const float* B, float* C, bool upper,
                            cudaStream_t st)
{
    if (R == 0) return cudaSuccess;
    int64_t gy = (R + SG_BM - 1) / SG_BM;
    if (gy > 65535) return cudaErrorInvalidValue;
    dim3 grid((Ncols + SG_BN - 1) / SG_BN, (unsigned)gy);
    const bool vec = K % 4 == 0 && Ncols % 4 == 0 &&
                     ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B) | reinterpret_cast<uintptr_t>(C)) & 15) == 0;
    auto kern = upper ? (vec ? sgemm_nn_kernel<true, true> : sgemm_nn_kernel<false, true>)
                      : (vec ? sgemm_nn_kernel<true, false> : sgemm_nn_kernel<false, false>);
    kern<<<grid, 256, 0, st>>>(R, Ncols, K, A, B, C);
    return cudaGetLastError();
}

}  // namespace fmc
