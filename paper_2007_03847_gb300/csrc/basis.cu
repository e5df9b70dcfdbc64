// Algorithm 1 step 2 (Eqs. kl, kle): increment basis of the truncated KL
// expansion, computed in FP64 on the GPU and rounded for the contraction.
//
// Brownian eigenbasis (FMC_BASIS_SINE):
//   phi[k][n] = c_k (sin(a_k t_{n+1}) - sin(a_k t_n)),  a_k = (k+1/2) pi / T,
//   c_k = sqrt(2T) / ((k+1/2) pi),  t_n = n T / Nt,   k = 0..K-1.
// Written without cancellation as a product,
//   phi[k][n] = 2 c_k cos(pi (2k+1)(2n+1) / (4 Nt)) sin(pi (2k+1) / (4 Nt)),
// with the argument of the cosine reduced exactly in integers modulo its period
// (8 Nt in units of pi / (4 Nt)) and evaluated by cospi / sinpi.
//
// The paper's basis of Eq. (klb2) (FMC_BASIS_COSINE), integrated over a step:
//   k = 0:  dt / sqrt(T)  (the constant mode 1/sqrt(T));
//   k >= 1: c_k (sin(a_k t_{n+1}) - sin(a_k t_n)), a_k = k pi / T, c_k = sqrt(2T)/(k pi)
//         = 2 c_k cos(pi k (2n+1) / (2 Nt)) sin(pi k / (2 Nt)),
// the cosine's argument reduced modulo 4 Nt (units of pi / (2 Nt)).
#include <cuda_bf16.h>

#include "fmc_common.cuh"
#include "kernels.cuh"

namespace fmc {

// An entry is (amplitude of k) x cos(pi m / P) x (sine of k) with an integer residue m:
// only P' distinct cosines for K Nt entries.  FP64 arithmetic is the bound (two FMA
// per SM and clock on this part), so the cosines of all residues are tabulated once
// per call (trig_table_kernel) and an entry costs two FP64 products, the residue kept
// by additions modulo the period along a thread's times.  Without the table (few
// entries, no room for it, the allocation-free reconstruction) a thread evaluates the
// cosine itself.  The
// operations per entry are the same either way, in the same order.
// Measured (GB300), split form: K = 200, Nt = 4000 148 -> 28 us; K = 100, Nt = 1000
// 32 -> 17 us, the table's 4 us included.
struct BasisArgs {
    int K, Nt, basis;
    double T;
    int forcing;           // the smooth form's forcing (below) instead of the increments
    const double* table;   // cosines by residue (by odd residue for the sine increments), then amplitude and
                           // sine of every k; or null
    int64_t cosines;       // entries of the table before the rows'
};

// The period of the cosine's argument in units of pi / den: den = period / 2.
__host__ __device__ inline int64_t basis_period(int Nt, int basis)
{
    return basis == FMC_BASIS_COSINE ? 4LL * Nt : 8LL * Nt;
}

// Entries of the table: all residues, or the odd ones (the sine increments' products
// of odd numbers).
static int64_t basis_table_entries(int Nt, int basis, int forcing)
{
    return (basis == FMC_BASIS_SINE && !forcing) ? 4LL * Nt : basis_period(Nt, basis);
}

int64_t basis_table_doubles(int K, int Nt, int basis, int forcing)
{
    return basis_table_entries(Nt, basis, forcing) + 2 * (int64_t)K;
}

__device__ __forceinline__ double basis_cos(int64_t m, int Nt, int basis)
{
    return cospi((double)m / (basis == FMC_BASIS_COSINE ? 2.0 * Nt : 4.0 * Nt));
}

// The forcing of the smooth form (Eq. eqkl as a random ODE): the time
// derivative of the basis function at the half-step times t = j T / (2 Nt),
// j = 0..2 Nt.  Brownian eigenbasis: sqrt(2/T) cos((k+1/2) pi t / T) =
// sqrt(2/T) cospi((2k+1) j / (4 Nt)), the argument reduced modulo 8 Nt; the
// paper's basis: 1/sqrt(T) (k = 0), sqrt(2/T) cospi(k j / (2 Nt)) (mod 4 Nt).
// What an entry of row k needs besides its cosine: value = (amp cos) sine (increments)
// or amp cos (forcing); the constant mode of the cosine basis has no cosine.
struct BasisRow {
    double amp, sine;
    bool flat;       // value = amp
    uint32_t odd;    // 2k+1 or k: the residue of time index j is odd * (2j+1) (increments) or odd * j
};

__device__ __forceinline__ BasisRow basis_row(const BasisArgs& a, int k)
{
    const double PI = 3.141592653589793238462643;
    BasisRow r;
    const bool cosine = a.basis == FMC_BASIS_COSINE;
    r.flat = cosine && k == 0;
    r.odd = cosine ? (uint32_t)k : 2u * (uint32_t)k + 1u;
    r.sine = 1.0;
    if (a.forcing) {
        r.amp = r.flat ? 1.0 / sqrt(a.T) : sqrt(2.0 / a.T);
        return r;
    }
    if (r.flat) {
        r.amp = sqrt(a.T) / (double)a.Nt;
    } else if (cosine) {
        const double c = sqrt(2.0 * a.T) / ((double)k * PI);
        r.amp = 2.0 * c;
        r.sine = sinpi((double)k / (2.0 * a.Nt));
    } else {
        const double c = 2.0 * sqrt(2.0 * a.T) / ((double)(2 * k + 1) * PI);
        r.amp = 2.0 * c;
        r.sine = sinpi((double)(2 * k + 1) / (4.0 * a.Nt));
    }
    return r;
}

// The table: the cosines, then (amplitude, sine) of every row.
__global__ void trig_table_kernel(BasisArgs a, int odd, double* __restrict__ table)
{
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e < a.cosines) {
        table[e] = basis_cos(odd ? 2 * e + 1 : e, a.Nt, a.basis);
    } else if (e - a.cosines < a.K) {
        const BasisRow r = basis_row(a, (int)(e - a.cosines));
        table[a.cosines + 2 * (e - a.cosines)] = r.amp;
        table[a.cosines + 2 * (e - a.cosines) + 1] = r.sine;
    }
}

// Row k with its FP64 constants from the table, where there is one.
__device__ __forceinline__ BasisRow basis_row_of(const BasisArgs& a, int k)
{
    if (!a.table) return basis_row(a, k);
    BasisRow r;
    r.flat = a.basis == FMC_BASIS_COSINE && k == 0;
    r.odd = a.basis == FMC_BASIS_COSINE ? (uint32_t)k : 2u * (uint32_t)k + 1u;
    r.amp = __ldg(a.table + a.cosines + 2 * (int64_t)k);
    r.sine = __ldg(a.table + a.cosines + 2 * (int64_t)k + 1);
    return r;
}

// x y mod P (32-bit arithmetic where the product allows it).
__device__ __forceinline__ int64_t mod_product(int64_t x, int64_t y, int64_t P)
{
    const int64_t m = x * y;
    if (m >> 32 == 0 && P >> 32 == 0) return (uint32_t)m % (uint32_t)P;
    return m % P;
}

__device__ __forceinline__ float basis_entry(const BasisArgs& a, const BasisRow& r, int64_t m)
{
    if (r.flat) return (float)r.amp;
    const double c = a.table ? __ldg(a.table + ((a.basis == FMC_BASIS_SINE && !a.forcing) ? m >> 1 : m))
                             : basis_cos(m, a.Nt, a.basis);
    return a.forcing ? (float)(r.amp * c) : (float)(r.amp * c * r.sine);
}

// The residue of row r at time index j, and the advance per `step` time indices.
__device__ __forceinline__ int64_t basis_residue(const BasisArgs& a, const BasisRow& r, int64_t j)
{
    return mod_product(r.odd, a.forcing ? j : 2 * j + 1, basis_period(a.Nt, a.basis));
}
__device__ __forceinline__ int64_t basis_advance(const BasisArgs& a, const BasisRow& r, int64_t step)
{
    return mod_product(r.odd, a.forcing ? step : 2 * step, basis_period(a.Nt, a.basis));
}

// FP32 [K][J] (J times; J contiguous): a CTA takes row k = blockIdx.y.
__global__ void __launch_bounds__(256) basis_f32_kernel(BasisArgs a, int J, float* __restrict__ phi)
{
    const int64_t P = basis_period(a.Nt, a.basis);
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    for (int k = blockIdx.y; k < a.K; k += gridDim.y) {
        const BasisRow r = basis_row_of(a, k);
        int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
        int64_t m = basis_residue(a, r, j);
        const int64_t dm = j + step < J ? basis_advance(a, r, step) : 0;
        for (; j < J; j += step) {
            phi[(int64_t)k * J + j] = basis_entry(a, r, m);
            m += dm;
            if (m >= P) m -= P;
        }
    }
}

// Time-major split BF16 for the tensor-core B operand: hi/lo [J][Kpad], zeros for
// k >= K.  A thread keeps its k and steps over times, a warp (32 k) per time.
__global__ void __launch_bounds__(256) basis_split_kernel(BasisArgs a, int J, int Kpad, __nv_bfloat16* __restrict__ hi,
                                                          __nv_bfloat16* __restrict__ lo)
{
    const int64_t P = basis_period(a.Nt, a.basis);
    const int times = (int)blockDim.x / 32;
    const int64_t step = (int64_t)gridDim.x * times;
    for (int k = blockIdx.y * 32 + threadIdx.x % 32; k < Kpad; k += gridDim.y * 32) {
        const bool real = k < a.K;
        const BasisRow r = basis_row_of(a, real ? k : 0);
        int64_t j = blockIdx.x * (int64_t)times + threadIdx.x / 32;
        int64_t m = basis_residue(a, r, j);
        const int64_t dm = j + step < J ? basis_advance(a, r, step) : 0;
        for (; j < J; j += step) {
            const float v = real ? basis_entry(a, r, m) : 0.f;
            const __nv_bfloat16 h = __float2bfloat16_rn(v);
            hi[j * Kpad + k] = h;
            if (lo) lo[j * Kpad + k] = __float2bfloat16_rn(v - __bfloat162float(h));
            m += dm;
            if (m >= P) m -= P;
        }
    }
}

// The table pays from some ten thousand entries on: filling it is a launch of its own
// (50 x 500 entries, FP32 result of 128 rows: 27 us with it, 25 without; 6 x 12000 split:
// 35 with it, 62 without).
constexpr int64_t BASIS_TABLE_MIN = 32768;

static cudaError_t basis_prepare(BasisArgs& a, double* table, int64_t entries, cudaStream_t st)
{
    a.table = nullptr;
    if (!table || entries < BASIS_TABLE_MIN) return cudaSuccess;
    a.cosines = basis_table_entries(a.Nt, a.basis, a.forcing);
    const int odd = a.basis == FMC_BASIS_SINE && !a.forcing;
    trig_table_kernel<<<(unsigned)((a.cosines + a.K + 63) / 64), 64, 0, st>>>(a, odd, table);
    a.table = table;
    return cudaGetLastError();
}

// Threads per block and entries per thread.  A thread's row constants and residue cost a
// few entries' work, so it takes up to eight entries once there are enough of them; and
// since a lone SM's FP64 pipe takes 16 cycles per warp instruction, small tables go to
// the SMs in blocks of 64 threads.  Measured (GB300, FP32 rows without the table, launches
// in a row; eight entries per thread in blocks of 256 -> now): 6 x 400 entries 12.4 ->
// 7.6 us, 60 x 4000 39 -> 25, 200 x 4000 70 either way.
struct BasisShape {
    int threads;
    int64_t entries;
};

static BasisShape basis_shape(int64_t entries, int sms)
{
    const int64_t e = entries / ((int64_t)sms * 128);
    return BasisShape{e < 8 ? 64 : 256, e < 1 ? 1 : (e > 8 ? 8 : e)};
}

static cudaError_t launch_f32(BasisArgs a, double* table, float* phi, int sms, cudaStream_t st)
{
    const int64_t J = a.forcing ? 2 * (int64_t)a.Nt + 1 : a.Nt;
    if (J > 2147483647LL) return cudaErrorInvalidValue;
    cudaError_t e = basis_prepare(a, table, a.K * J, st);
    if (e != cudaSuccess) return e;
    const BasisShape b = basis_shape(a.K * J, sms);
    const int gy = a.K < 65535 ? a.K : 65535;
    const int64_t per = b.threads * b.entries;
    int64_t gx = (J + per - 1) / per;
    const int64_t cap = ((int64_t)sms * 16 + gy - 1) / gy;
    if (gx > cap) gx = cap;
    basis_f32_kernel<<<dim3((unsigned)gx, (unsigned)gy), b.threads, 0, st>>>(a, (int)J, phi);
    return cudaGetLastError();
}

static cudaError_t launch_split(BasisArgs a, double* table, int Kpad, void* hi, void* lo, int sms, cudaStream_t st)
{
    const int64_t J = a.forcing ? 2 * (int64_t)a.Nt + 1 : a.Nt;
    if (J > 2147483647LL) return cudaErrorInvalidValue;
    cudaError_t e = basis_prepare(a, table, a.K * J, st);
    if (e != cudaSuccess) return e;
    const BasisShape b = basis_shape(Kpad * J, sms);
    const int ky = Kpad / 32;
    const int gy = ky < 65535 ? ky : 65535;
    const int64_t per = b.threads / 32 * b.entries;
    int64_t gx = (J + per - 1) / per;
    const int64_t cap = ((int64_t)sms * 16 + gy - 1) / gy;
    if (gx > cap) gx = cap;
    basis_split_kernel<<<dim3((unsigned)gx, (unsigned)gy), b.threads, 0, st>>>(a, (int)J, Kpad, (__nv_bfloat16*)hi,
                                                                              (__nv_bfloat16*)lo);
    return cudaGetLastError();
}

cudaError_t launch_forcing_split(int K, int Nt, double T, int basis, int Kpad, double* table, void* hi, void* lo,
                                 int sms, cudaStream_t st)
{
    return launch_split(BasisArgs{K, Nt, basis, T, 1, nullptr, 0}, table, Kpad, hi, lo, sms, st);
}

cudaError_t launch_forcing_f32(int K, int Nt, double T, int basis, double* table, float* phi, int sms, cudaStream_t st)
{
    return launch_f32(BasisArgs{K, Nt, basis, T, 1, nullptr, 0}, table, phi, sms, st);
}

cudaError_t launch_basis_f32(int K, int Nt, double T, int basis, double* table, float* phi, int sms, cudaStream_t st)
{
    return launch_f32(BasisArgs{K, Nt, basis, T, 0, nullptr, 0}, table, phi, sms, st);
}

cudaError_t launch_basis_split(int K, int Nt, double T, int basis, int Kpad, double* table, void* hi, void* lo,
                               int sms, cudaStream_t st)
{
    return launch_split(BasisArgs{K, Nt, basis, T, 0, nullptr, 0}, table, Kpad, hi, lo, sms, st);
}

}  // namespace fmc
