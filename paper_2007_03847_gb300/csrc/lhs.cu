// Algorithm 1 step 1 / Section IV-B: Latin hypercube sampling of the M = d*K
// KL coefficients on the GPU.  The design is stateless (a keyed Feistel
// permutation per dimension), so any sub-range of the N rows is produced
// bit-identically without sorting or communication.
#include <cuda_bf16.h>

#include <cmath>

#include "fmc_common.cuh"
#include "kernels.cuh"
#include "lhs_feistel.cuh"

namespace fmc {

constexpr int DESIGN_SMEM_MAX = 224 * 1024;

// ---------------------------------------------------------------------------
// design_kernel: the design's values of a tile of positions x samples.
//
// What bounds it: integer issue.  Computed from its definition, an entry costs
// seven Philox calls (six Feistel rounds and the uniform), and a domain 4^h above
// N repeats the six until the value falls below N (cycle walking).  But a round
// function takes its argument from h bits only, so per dimension it has 2^h
// values: a CTA tabulates the 6 x 2^h of its dimensions in shared memory (the
// masked Philox words, so the permutation is the same bit for bit) and a round
// becomes one lookup.  Tables pay from about 2^h rows per CTA on; the tile takes
// up to 16 x 2^h.
//
// Layout: a thread keeps one position (column) and steps over rows, with DB
// neighbouring positions in neighbouring lanes (16 bytes of a row; the rest of a
// sector meets them in L2), and no index division is left in the loop.  Strata go
// through a short per-thread list in shared memory: walking lanes take their next
// row as soon as their value is found instead of waiting for the warp's longest
// walk, and the list is read transposed where strata themselves are stored or
// loaded (their rows run along the samples).
//
// Measured (GB300, launches in a row): 65536 x 600 values and strata 735 -> 308 us
// (entries computed one by one from the definition before; 1 TB/s of output, the
// uniform's Philox call and the two branches of the inverse CDF now take the issue
// slots); the split-BF16 rows of 19001 x 2400 (domain 4^8, 3.4 walks per entry) 6.98 ->
// 0.60 ms.  With 16 positions per CTA (8 with uint16 tables) these took 361 us and
// 0.69 ms, the tables' filling being four times as long, and few columns left lanes
// idle: 2^20 x 20 by simple random sampling 179 us (one by one 125, now 115),
// 4.2e6 x 4 by the definition 4.61 ms (2.93, 1.37), 2^20 x 1 325 us (25, 23).
// ---------------------------------------------------------------------------
enum { PERM_NONE = 0, PERM_DIRECT, PERM_TAB8, PERM_TAB16, PERM_GIVEN };
enum { OUT_F32 = 0, OUT_SPLIT, OUT_SCORE };

template <int PERM, int DBN>
struct DesignTile {
    static constexpr int THREADS = PERM == PERM_TAB16 ? 512 : 256;
    static constexpr int DB = DBN;  // positions per CTA
    static constexpr int RPI = THREADS / DB;                 // rows per pass of the CTA
    static constexpr int LCAP = PERM == PERM_TAB16 ? 4 : 16; // list entries per thread
    static constexpr int SUB = RPI * LCAP;                   // rows per list filling
    static constexpr int LIST_BYTES = SUB * (DB + 1) * 4;
};

struct DesignArgs {
    uint32_t k0s, k1s, N;
    int64_t k0, count;
    int cols;          // positions per row: M, or d Ks with K..Ks-1 of every group zero
    int K, Ks;         // OUT_SPLIT
    int mode, h;
    uint32_t mask;
    float rcp;         // see normal_from_fraction
    int walk;          // N < 4^h
    int npos;          // position blocks
    int64_t rows;      // rows per CTA
    float* zeta;       // OUT_F32 / OUT_SCORE [count][cols], may be null (strata only)
    __nv_bfloat16 *hi, *lo;
    uint32_t* strata;            // [M][count] out, or null
    const uint32_t* strata_in;   // PERM_GIVEN: [M][N]
    const double *score, *mean;  // OUT_SCORE: a(s) and its mean
};

template <int PERM>
__device__ __forceinline__ uint32_t feistel_round(const void* tab, uint32_t R, int r, const DesignArgs& a, uint32_t dim)
{
    if constexpr (PERM == PERM_TAB8)
        return static_cast<const uint8_t*>(tab)[((uint32_t)r << a.h) + R];
    else if constexpr (PERM == PERM_TAB16)
        return static_cast<const uint16_t*>(tab)[((uint32_t)r << a.h) + R];
    else
        return philox4x32_10(U4{R, dim, 1u + (uint32_t)r, 0u}, a.k0s, a.k1s).x & a.mask;
}

// One application of the Feistel network (feistel() of lhs_feistel.cuh).
template <int PERM>
__device__ __forceinline__ uint32_t permute(const void* tab, uint32_t x, const DesignArgs& a, uint32_t dim)
{
    uint32_t L = (x >> a.h) & a.mask, R = x & a.mask;
#pragma unroll
    for (int r = 0; r < kFeistelRounds; ++r) {
        const uint32_t n = L ^ feistel_round<PERM>(tab, R, r, a, dim);
        L = R;
        R = n;
    }
    return (L << a.h) | R;
}

template <int PERM, int OUT, int DB>
__global__ void __launch_bounds__(DesignTile<PERM, DB>::THREADS) design_kernel(const DesignArgs a)
{
    using T = DesignTile<PERM, DB>;
    extern __shared__ __align__(16) unsigned char dsm[];
    uint32_t* list = reinterpret_cast<uint32_t*>(dsm);
    unsigned char* tabs = dsm + T::LIST_BYTES;
    const int tid = threadIdx.x;
    const int dc = tid % T::DB, q = tid / T::DB;
    const int pb = (int)(blockIdx.x % (unsigned)a.npos);
    const int64_t j0 = (int64_t)(blockIdx.x / (unsigned)a.npos) * a.rows;
    const int64_t j1 = j0 + a.rows < a.count ? j0 + a.rows : a.count;
    const int pos = pb * T::DB + dc;
    // the dimension of this thread's position (split rows: groups of Ks, K of them real)
    uint32_t dim = (uint32_t)pos;
    bool real = pos < a.cols;
    if (OUT == OUT_SPLIT) {
        const int w = pos / a.Ks, kk = pos - w * a.Ks;
        dim = (uint32_t)(w * a.K + kk);
        real = real && kk < a.K;
    }
    const void* tab = nullptr;
    if constexpr (PERM == PERM_TAB8 || PERM == PERM_TAB16) {
        // the CTA's tables: [DB][6][2^h]
        constexpr int EB = PERM == PERM_TAB8 ? 1 : 2;
        const int per = kFeistelRounds << a.h;
        for (int e = q; e < per; e += T::RPI) {
            uint32_t v = 0;
            if (real)
                v = philox4x32_10(U4{(uint32_t)e & a.mask, dim, 1u + ((uint32_t)e >> a.h), 0u}, a.k0s, a.k1s).x & a.mask;
            if (EB == 1)
                tabs[dc * per + e] = (uint8_t)v;
            else
                reinterpret_cast<uint16_t*>(tabs)[dc * per + e] = (uint16_t)v;
        }
        __syncthreads();
        tab = tabs + (size_t)dc * per * EB;
    }
    for (int64_t jb = j0; jb < j1; jb += T::SUB) {
        const int nrow = j1 - jb < T::SUB ? (int)(j1 - jb) : T::SUB;  // rows of this filling
        const int mine = q < nrow ? (nrow - q + T::RPI - 1) / T::RPI : 0;
        uint32_t* my = list + q * (T::DB + 1) + dc;  // entry i at my[i * RPI * (DB + 1)]
        constexpr int LS = T::RPI * (T::DB + 1);
        const uint32_t kb = (uint32_t)(a.k0 + jb) + (uint32_t)q;
        if constexpr (PERM == PERM_GIVEN) {
            // strata_in rows run along the samples: read them so, transposed into the list
            __syncthreads();
            for (int e = tid; e < T::DB * T::SUB; e += T::THREADS) {
                const int c = e / T::SUB, row = e % T::SUB;
                const int p2 = pb * T::DB + c;
                uint32_t dim2 = (uint32_t)p2;
                bool real2 = p2 < a.cols;
                if (OUT == OUT_SPLIT) {
                    const int w = p2 / a.Ks, kk = p2 - w * a.Ks;
                    dim2 = (uint32_t)(w * a.K + kk);
                    real2 = real2 && kk < a.K;
                }
                if (real2 && row < nrow)
                    list[row * (T::DB + 1) + c] = a.strata_in[(int64_t)dim2 * a.N + a.k0 + jb + row];
            }
            __syncthreads();
        } else if constexpr (PERM != PERM_NONE) {
            if (a.walk) {
                int i = 0;
                uint32_t y = kb;
                while (real && i < mine) {
                    y = permute<PERM>(tab, y, a, dim);
                    if (y < a.N) {
                        my[i * LS] = y;
                        ++i;
                        y = kb + (uint32_t)(i * T::RPI);
                    }
                }
            } else if (real) {
#pragma unroll 2
                for (int i = 0; i < mine; ++i) my[i * LS] = permute<PERM>(tab, kb + (uint32_t)(i * T::RPI), a, dim);
            }
        } else if (a.strata) {
            for (int i = 0; i < mine; ++i) my[i * LS] = kb + (uint32_t)(i * T::RPI);  // (no permutation: s = k)
        }
        if (pos < a.cols && (OUT != OUT_F32 || a.zeta)) {
#pragma unroll 2
            for (int i = 0; i < mine; ++i) {
                const uint32_t k = kb + (uint32_t)(i * T::RPI);
                const int64_t o = (jb + q + i * T::RPI) * a.cols + pos;
                if constexpr (OUT == OUT_SCORE) {
                    a.zeta[o] = (float)(a.score[my[i * LS]] - *a.mean);
                } else {
                    float z = 0.f;
                    if (real) {
                        if (PERM == PERM_NONE) {
                            const uint32_t r = philox4x32_10(U4{k, dim, 0u, 0u}, a.k0s, a.k1s).x;
                            z = normal_from_fraction(2ull * r + 1ull, 1u, 0x1p-32f);
                        } else {
                            const uint32_t s = my[i * LS];
                            uint64_t num2 = ((uint64_t)s << 33) + (1ull << 32);
                            if (a.mode != FMC_LHS_MIDPOINT) {
                                const uint32_t r = philox4x32_10(U4{k, dim, 0u, 0u}, a.k0s, a.k1s).x;
                                num2 = ((uint64_t)s << 33) + 2ull * r + 1ull;
                            }
                            z = normal_from_fraction(num2, a.N, a.rcp);
                        }
                    }
                    if constexpr (OUT == OUT_F32) {
                        a.zeta[o] = z;
                    } else {
                        const __nv_bfloat16 zh = __float2bfloat16_rn(z);
                        a.hi[o] = zh;
                        if (a.lo) a.lo[o] = __float2bfloat16_rn(z - __bfloat162float(zh));
                    }
                }
            }
        }
        if (OUT == OUT_F32 && a.strata) {
            __syncthreads();
            for (int e = tid; e < T::DB * T::SUB; e += T::THREADS) {
                const int c = e / T::SUB, row = e % T::SUB;
                const int p2 = pb * T::DB + c;
                if (p2 < a.cols && row < nrow) a.strata[(int64_t)p2 * a.count + jb + row] = list[row * (T::DB + 1) + c];
            }
            __syncthreads();
        }
    }
}

template <int PERM, int OUT, int DB>
static cudaError_t launch_design_db(DesignArgs& a, int sms, cudaStream_t st)
{
    using T = DesignTile<PERM, DB>;
    constexpr bool TAB = PERM == PERM_TAB8 || PERM == PERM_TAB16;
    a.npos = (a.cols + T::DB - 1) / T::DB;
    // rows per CTA: four CTAs per SM in all (eight where no walks need evening out: 2^20 x 8
    // by simple random sampling 54 -> 45 us), but 2 .. 16 rows per table entry where there
    // are tables (their filling is at most three Philox calls per entry, at most 3/8 for
    // large designs), and whole list fillings (whole passes below one)
    const bool even = PERM == PERM_NONE || (PERM == PERM_DIRECT && !a.walk);
    const int64_t ctas = (even ? 8 : 4) * (int64_t)sms;
    int64_t rows = (a.count * a.npos + ctas - 1) / ctas;
    const int64_t lo = TAB ? (int64_t)2 << a.h : 1, hi = TAB ? (int64_t)16 << a.h : (int64_t)1 << 14;
    rows = rows < lo ? lo : (rows > hi ? hi : rows);
    const int64_t unit = rows < T::SUB ? T::RPI : T::SUB;
    rows = (rows + unit - 1) / unit * unit;
    while ((a.count + rows - 1) / rows * a.npos > 2147483647LL) rows *= 2;
    a.rows = rows;
    const int smem = T::LIST_BYTES + (TAB ? T::DB * (kFeistelRounds << a.h) * (PERM == PERM_TAB8 ? 1 : 2) : 0);
    auto kern = design_kernel<PERM, OUT, DB>;
    if (smem > 48 * 1024) {
        // process-wide attribute: always the same bound (launches may race on it)
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, DESIGN_SMEM_MAX);
        if (e != cudaSuccess) return e;
    }
    const int64_t grid = (a.count + rows - 1) / rows * a.npos;
    kern<<<(unsigned)grid, T::THREADS, smem, st>>>(a);
    return cudaGetLastError();
}

// Four positions per CTA, or one where there are fewer than four (idle lanes).
template <int PERM, int OUT>
static cudaError_t launch_design_t(DesignArgs& a, int sms, cudaStream_t st)
{
    return a.cols < 4 ? launch_design_db<PERM, OUT, 1>(a, sms, st) : launch_design_db<PERM, OUT, 4>(a, sms, st);
}

// Whether tables pay for a design that fits them (h <= 11).  Blocks of 2^(h+1) rows at
// least repay the filling; where they are fewer than four per SM, the threads' chains
// decide: the filling and the lookups against the rounds by definition of fewer rows per
// thread, in Philox calls (the uniform and the inverse CDF are worth three, a lookup half a
// call), the definition a fifth off since its SMs are the fuller.  With and without tables
// (us, launches in a row): 30000 rows of a 2^22-sample design, 20 columns, 47 and 15; 60000
// rows of 2^18, 10 columns, 23 and 16; 65536 x 20 25 and 27.
static bool tables_pay(const DesignArgs& a, int sms)
{
    const int64_t least = (int64_t)2 << a.h;
    if (a.count < least) return false;
    const int db = a.cols < 4 ? 1 : 4, threads = a.h <= 8 ? 256 : 512;
    const int64_t npos = (a.cols + db - 1) / db, rows = (a.count * npos + 4 * sms - 1) / (4 * (int64_t)sms);
    if (rows >= least) return true;
    auto passes = [db](int64_t r, int t) { return (double)((r * db + t - 1) / t); };
    // (a warp's lanes wait for the longest of their walks: the largest of 32 geometric numbers)
    const double stay = (double)a.N / (double)((uint64_t)1 << (2 * a.h));
    const double walk = a.walk ? 0.5 - std::log(32.0) / std::log1p(-stay) : 1.0;
    const double table = kFeistelRounds * (double)((int64_t)db << a.h) / threads + 3.5 * passes(least, threads);
    return 0.8 * (kFeistelRounds * walk + 3.0) * passes(rows, 256) >= table;
}

// The rule: tables while they fit (uint8 up to h = 8, 6 KB; uint16 up to h = 11, 96 KB) and
// pay; the rounds from their definition above (more than 2^22 samples) and for short blocks
// of a large design; no permutation for simple random sampling.
template <int OUT>
static cudaError_t launch_design(DesignArgs& a, int sms, cudaStream_t st)
{
    if (a.count == 0) return cudaSuccess;
    if (a.strata_in) return launch_design_t<PERM_GIVEN, OUT>(a, sms, st);
    if (a.mode == FMC_SRS) return launch_design_t<PERM_NONE, OUT>(a, sms, st);
    if (a.h <= 11 && tables_pay(a, sms)) {
        if (a.h <= 8) return launch_design_t<PERM_TAB8, OUT>(a, sms, st);
        return launch_design_t<PERM_TAB16, OUT>(a, sms, st);
    }
    return launch_design_t<PERM_DIRECT, OUT>(a, sms, st);
}

static DesignArgs design_args(uint64_t seed, int64_t N, int64_t k0, int64_t count, int cols, int mode)
{
    const FeistelShape f = feistel_shape(N);
    DesignArgs a{};
    a.k0s = (uint32_t)seed;
    a.k1s = (uint32_t)(seed >> 32);
    a.N = (uint32_t)N;
    a.k0 = k0;
    a.count = count;
    a.cols = cols;
    a.mode = mode;
    a.h = f.h;
    a.mask = f.mask;
    a.walk = f.walk;
    a.rcp = (N & (N - 1)) == 0 ? 0x1p-32f / (float)N : 0.f;
    return a;
}

// The paper's traditional Monte Carlo (Section V-B, Eq. distito): increments
// dW[s][w][n] = sqrt(dt) em_normal(seed, k0 + s, w, n) of samples k0..k0+count-1.
__global__ void em_increments_kernel(uint32_t k0s, uint32_t k1s, int64_t k0, int64_t count, int d, int Nt,
                                     float sqdt, float* __restrict__ dW)
{
    int64_t total = count * (int64_t)d * Nt;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        int64_t sw = t / Nt;
        int n = (int)(t - sw * Nt);
        int64_t s = sw / d;
        int w = (int)(sw - s * d);
        dW[t] = sqdt * em_normal((uint32_t)(k0 + s), w, n, k0s, k1s);
    }
}

static int grid_for(int64_t total, int block, int sms)
{
    int64_t g = (total + block - 1) / block;
    int64_t cap = (int64_t)sms * 32;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (int)g;
}

cudaError_t launch_lhs_f32(uint64_t seed, int64_t N, int64_t k0, int64_t count, int M, int mode, float* zeta,
                           uint32_t* strata, int sms, cudaStream_t st)
{
    DesignArgs a = design_args(seed, N, k0, count, M, mode);
    a.zeta = zeta;
    a.strata = strata;
    return launch_design<OUT_F32>(a, sms, st);
}

cudaError_t launch_lhs_split(uint64_t seed, int64_t N, int64_t k0, int64_t count, int d, int K, int mode,
                             const uint32_t* strata, void* hi, void* lo, int sms, cudaStream_t st)
{
    const int Ks = round_up(K, 8);
    DesignArgs a = design_args(seed, N, k0, count, d * Ks, mode);
    a.K = K;
    a.Ks = Ks;
    a.hi = static_cast<__nv_bfloat16*>(hi);
    a.lo = static_cast<__nv_bfloat16*>(lo);
    a.strata_in = strata;
    return launch_design<OUT_SPLIT>(a, sms, st);
}

cudaError_t launch_strata_values(uint64_t seed, int64_t N, int64_t k0, int64_t count, int M, int mode,
                                 const uint32_t* strata, float* zeta, int sms, cudaStream_t st)
{
    DesignArgs a = design_args(seed, N, k0, count, M, mode);
    a.zeta = zeta;
    a.strata_in = strata;
    return launch_design<OUT_F32>(a, sms, st);
}

cudaError_t launch_design_scores(uint64_t seed, int64_t N, int M, const double* score, const double* mean, float* R,
                                 int sms, cudaStream_t st)
{
    DesignArgs a = design_args(seed, N, 0, N, M, FMC_LHS);
    a.zeta = R;
    a.score = score;
    a.mean = mean;
    return launch_design<OUT_SCORE>(a, sms, st);
}

cudaError_t launch_em_increments(uint64_t seed, int64_t k0, int64_t count, int d, int Nt, double dt, float* dW,
                                 int sms, cudaStream_t st)
{
    if (count == 0) return cudaSuccess;
    int64_t total = count * (int64_t)d * Nt;
    em_increments_kernel<<<grid_for(total, 256, sms), 256, 0, st>>>((uint32_t)seed, (uint32_t)(seed >> 32), k0, count,
                                                                    d, Nt, (float)sqrt(dt), dW);
    return cudaGetLastError();
}

}  // namespace fmc
