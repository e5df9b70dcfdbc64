// Section IV-B step 2 on the GPU: a permutation of the primary sampling matrix
// that minimises the correlation between its columns.  The paper names a
// Cholesky-based method without giving it; this is the rank method of Iman and
// Conover (1982) with the identity as target correlation:
//   R[k][i] = a(pi_i(k)),  a(s) = Phi^-1((s + 1) / (N + 1)) - mean  (centred
//            van der Waerden scores paired by the design's own permutations),
//   T = R^T R / (N var a) = Q Q^T,   R* = R Q^-T,
//   pi'_i(k) = rank of R*[k][i] in column i (ascending, ties by sample index),
// and every sample keeps its uniform inside its new stratum.
//
// Kernels: the score table (FP64, one value per stratum), the centred score
// matrix [N][M] (FP32), its Gram matrix (FP32 tiles summed in FP64), a blocked
// Cholesky factorisation and triangular inverse in FP32 (T is within O(1/sqrt N)
// of the identity), R* by the FP32 GEMM, the per-column ranks by a segmented
// radix sort (CUB), and the design values from the new strata.
#include <cub/device/device_segmented_radix_sort.cuh>

#include "fmc_common.cuh"
#include "kernels.cuh"

namespace fmc {

// a(s) = Phi^-1((s + 1) / (N + 1)) in FP64, s < N; the tails through erfcinv so
// that the smallest probabilities keep their relative accuracy.
__global__ void ic_score_table_kernel(uint32_t N, double* __restrict__ a)
{
    for (uint32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < N; s += gridDim.x * blockDim.x) {
        const double p = ((double)s + 1.0) / ((double)N + 1.0);
        const double SQRT2 = 1.4142135623730951;
        double z;
        if (p < 0.25)
            z = -SQRT2 * erfcinv(2.0 * p);
        else if (p > 0.75)
            z = SQRT2 * erfcinv(2.0 * (((double)N - (double)s) / ((double)N + 1.0)));
        else
            z = SQRT2 * erfinv(2.0 * p - 1.0);
        a[s] = z;
    }
}

// mean and sum of squares about it of the N scores (one CTA of 1024 threads)
__global__ void ic_score_moments_kernel(uint32_t N, const double* __restrict__ a, double* __restrict__ out)
{
    __shared__ double red[1024];
    double s = 0.0;
    for (uint32_t i = threadIdx.x; i < N; i += blockDim.x) s += a[i];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    const double mean = red[0] / (double)N;
    __syncthreads();
    double q = 0.0;
    for (uint32_t i = threadIdx.x; i < N; i += blockDim.x) q += (a[i] - mean) * (a[i] - mean);
    red[threadIdx.x] = q;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[0] = mean;
        out[1] = red[0];
    }
}

// G = R^T R (FP64 [M][M], zeroed by the caller): a CTA of 256 threads sums a
// 64 x 64 tile over a range of IC_GRAM_ROWS rows in FP32 (4 x 4 outputs per
// thread, rows staged through shared memory) and adds it into G in FP64.
constexpr int IC_GT = 64, IC_GK = 32, IC_GRAM_ROWS = 1024;

__global__ void __launch_bounds__(256) ic_gram_kernel(int64_t N, int M, const float* __restrict__ R,
                                                      double* __restrict__ G)
{
    __shared__ float As[IC_GK][IC_GT];
    __shared__ float Bs[IC_GK][IC_GT];
    const int bi = blockIdx.x, bj = blockIdx.y;
    if (bj > bi) return;  // lower triangle of tiles; mirrored below
    const int i0 = bi * IC_GT, j0 = bj * IC_GT;
    const int64_t r0 = (int64_t)blockIdx.z * IC_GRAM_ROWS;
    const int64_t r1 = (r0 + IC_GRAM_ROWS < N) ? r0 + IC_GRAM_ROWS : N;
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    float acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;
    for (int64_t k0 = r0; k0 < r1; k0 += IC_GK) {
        for (int e = threadIdx.x; e < IC_GK * IC_GT; e += 256) {
            const int kk = e / IC_GT, c = e % IC_GT;
            const int64_t k = k0 + kk;
            As[kk][c] = (k < r1 && i0 + c < M) ? R[k * M + i0 + c] : 0.f;
            Bs[kk][c] = (k < r1 && j0 + c < M) ? R[k * M + j0 + c] : 0.f;
        }
        __syncthreads();
#pragma unroll 8
        for (int kk = 0; kk < IC_GK; ++kk) {
            float av[4], bv[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) av[a] = As[kk][ty * 4 + a];
#pragma unroll
            for (int b = 0; b < 4; ++b) bv[b] = Bs[kk][tx * 4 + b];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] = fmaf(av[a], bv[b], acc[a][b]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int i = i0 + ty * 4 + a, j = j0 + tx * 4 + b;
            if (i < M && j <= i) atomicAdd(&G[(int64_t)i * M + j], (double)acc[a][b]);
        }
}

// Cholesky factor Q of T = corr(R) (T_ij = G_ij / sqrt(G_ii G_jj)) in place in the
// lower triangle of A [M][M] (FP32), in panels of IC_NB columns: the panel kernel
// solves the panel's rows below its diagonal block, the update kernel takes the
// rank-IC_NB update off the trailing triangle and factors the next diagonal block.  Every entry takes its updates one column at a time in column
// order (a right-looking elimination), so the factor does not depend on the panel
// width.  (One CTA walking the columns of the whole matrix in memory, three barriers
// each, and the inverse by one thread per column took 19 of the 21.6 ms of a
// 16384 x 600 permutation; factor and inverse now take 0.8 of 1.97 ms.)
constexpr int IC_MAX_M = 4096;
constexpr int IC_NB = 32;

__global__ void ic_corr_kernel(int M, const double* __restrict__ G, float* __restrict__ A, int* __restrict__ ok)
{
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e == 0) *ok = 1;
    if (e >= (int64_t)M * M) return;
    const int i = (int)(e / M), j = (int)(e % M);
    float v = 0.f;
    if (i == j)
        v = 1.f;
    else if (j < i)
        v = (float)(G[e] / sqrt(G[(int64_t)i * M + i] * G[(int64_t)j * M + j]));
    A[e] = v;
}

// The diagonal block at p0, factored in place by one warp (lane = row).  *ok = 0 if a
// pivot is not positive (T not positive definite).
__device__ void ic_factor_block(int M, int p0, float* __restrict__ A, int* __restrict__ ok)
{
    const int lane = threadIdx.x, nb = M - p0 < IC_NB ? M - p0 : IC_NB;
    float* row = A + (int64_t)(p0 + lane) * M + p0;
    float r[IC_NB];
#pragma unroll
    for (int j = 0; j < IC_NB; ++j) r[j] = (lane < nb && j <= lane) ? row[j] : 0.f;
    bool good = true;
#pragma unroll
    for (int j = 0; j < IC_NB; ++j) {
        const float d = __shfl_sync(0xffffffffu, r[j], j);
        if (j < nb && !(d > 0.f)) good = false;
        const float piv = d > 0.f ? sqrtf(d) : 1.f;
        r[j] = lane == j ? piv : r[j] / piv;
#pragma unroll
        for (int k = j + 1; k < IC_NB; ++k) {
            const float lk = __shfl_sync(0xffffffffu, r[j], k);  // Q[k][j]
            if (k <= lane) r[k] = fmaf(-r[j], lk, r[k]);
        }
    }
#pragma unroll
    for (int j = 0; j < IC_NB; ++j)
        if (lane < nb && j <= lane) row[j] = r[j];
    if (lane == 0 && !good) *ok = 0;
}

__global__ void __launch_bounds__(32) ic_first_block_kernel(int M, float* __restrict__ A, int* __restrict__ ok)
{
    ic_factor_block(M, 0, A, ok);
}

// Columns p0 .. p0 + IC_NB - 1 of the rows past the (factored) diagonal block, one
// row per thread.
__global__ void __launch_bounds__(128) ic_panel_kernel(int M, int p0, float* __restrict__ A)
{
    __shared__ float D[IC_NB][IC_NB + 1];
    const int tid = threadIdx.x;
    for (int e = tid; e < IC_NB * IC_NB; e += 128) {
        const int i = e / IC_NB, j = e % IC_NB;
        D[i][j] = A[(int64_t)(p0 + i) * M + p0 + j];
    }
    __syncthreads();
    const int i = p0 + IC_NB + blockIdx.x * 128 + tid;
    if (i >= M) return;
    float r[IC_NB];
    float* row = A + (int64_t)i * M + p0;
#pragma unroll
    for (int j = 0; j < IC_NB; ++j) r[j] = row[j];
#pragma unroll
    for (int j = 0; j < IC_NB; ++j) {
        r[j] = r[j] / D[j][j];
#pragma unroll
        for (int k = j + 1; k < IC_NB; ++k) r[k] = fmaf(-r[j], D[k][j], r[k]);
    }
#pragma unroll
    for (int j = 0; j < IC_NB; ++j) row[j] = r[j];
}

// A[i][k] -= sum over the panel's columns j, in order, of Q[i][j] Q[k][j], for
// i >= k >= p1 = p0 + IC_NB: one CTA per 64 x 64 tile, 4 x 4 entries per thread.  The
// CTA of the first tile then factors the next diagonal block (which it alone wrote).
__global__ void __launch_bounds__(256) ic_update_kernel(int M, int p0, float* __restrict__ A, int* __restrict__ ok)
{
    if (blockIdx.y > blockIdx.x) return;  // the lower triangle of tiles
    __shared__ float Li[IC_NB][64 + 1], Lk[IC_NB][64 + 1];
    const int p1 = p0 + IC_NB, i0 = p1 + blockIdx.x * 64, k0 = p1 + blockIdx.y * 64;
    for (int e = threadIdx.x; e < 64 * IC_NB; e += 256) {
        const int r = e / IC_NB, j = e % IC_NB;
        Li[j][r] = i0 + r < M ? A[(int64_t)(i0 + r) * M + p0 + j] : 0.f;
        Lk[j][r] = k0 + r < M ? A[(int64_t)(k0 + r) * M + p0 + j] : 0.f;
    }
    __syncthreads();
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    float acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int i = i0 + ty + 16 * a, k = k0 + tx + 16 * b;
            acc[a][b] = (i < M && k <= i) ? A[(int64_t)i * M + k] : 0.f;
        }
#pragma unroll 8
    for (int j = 0; j < IC_NB; ++j) {
        float lk[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) lk[b] = Lk[j][tx + 16 * b];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const float li = -Li[j][ty + 16 * a];
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[a][b] = fmaf(li, lk[b], acc[a][b]);
        }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int i = i0 + ty + 16 * a, k = k0 + tx + 16 * b;
            if (i < M && k <= i) A[(int64_t)i * M + k] = acc[a][b];
        }
    if (blockIdx.x == 0) {
        __syncthreads();
        if (threadIdx.x < 32) ic_factor_block(M, p1, A, ok);
    }
}

// B = Q^-T [M][M] (row-major): row c of B is the solution w of Q w = e_c by forward
// substitution, w_r = -(sum over k = c .. r-1, in order, of Q[r][k] w_k) / Q[r][r].  A CTA
// takes IC_CB rows c and walks the blocks of IC_NB columns k: one warp per row
// solves the block's triangle (lane = r), then all threads add the block's terms to
// the sums of the later r, kept in shared memory, so the terms of every sum still
// come one by one in the order of k.  (0.12 ms at M = 600.)
constexpr int IC_CB = 4;

__global__ void __launch_bounds__(256) ic_inverse_kernel(int M, const float* __restrict__ Q, float* __restrict__ B)
{
    extern __shared__ float V[];  // [IC_CB][M]: the sums
    __shared__ float wv[IC_CB][IC_NB];
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int c0 = blockIdx.x * IC_CB;
    for (int e = tid; e < IC_CB * M; e += 256) V[e] = 0.f;
    for (int e = tid; e < IC_CB * M; e += 256) {
        const int c = c0 + e / M, r = e % M;
        if (c < M && r < c) B[(int64_t)c * M + r] = 0.f;
    }
    __syncthreads();
    for (int r0 = c0 / IC_NB * IC_NB; r0 < M; r0 += IC_NB) {
        const int nb = M - r0 < IC_NB ? M - r0 : IC_NB;
        if (warp < IC_CB) {
            const int c = c0 + warp, r = r0 + lane;
            const bool in = c < M && lane < nb;
            float q[IC_NB];  // Q[r][r0 ..]
#pragma unroll
            for (int s = 0; s < IC_NB; ++s) q[s] = (in && s <= lane) ? Q[(int64_t)r * M + r0 + s] : 0.f;
            float v = in ? V[warp * M + r] : 0.f, mine = 0.f;
            const float dia = in ? Q[(int64_t)r * M + r] : 1.f;
            const float rec = 1.f / dia;  // w_c itself
#pragma unroll
            for (int s = 0; s < IC_NB; ++s) {
                const float cand = r < c ? 0.f : (r == c ? rec : -v / dia);
                const float ws = __shfl_sync(0xffffffffu, cand, s);
                if (lane == s) mine = ws;
                if (lane > s) v = fmaf(q[s], ws, v);
            }
            wv[warp][lane] = mine;
            if (in && r >= c) B[(int64_t)c * M + r] = mine;
        }
        __syncthreads();
        for (int r = r0 + IC_NB + tid; r < M; r += 256) {
            float q[IC_NB];
#pragma unroll
            for (int s = 0; s < IC_NB; ++s) q[s] = Q[(int64_t)r * M + r0 + s];
#pragma unroll
            for (int u = 0; u < IC_CB; ++u) {
                float v = V[u * M + r];
#pragma unroll
                for (int s = 0; s < IC_NB; ++s) v = fmaf(q[s], wv[u][s], v);
                V[u * M + r] = v;
            }
        }
        __syncthreads();
    }
}

// keys for the per-column ranking: column i of R* [N][M] as order-preserving
// unsigned integers, transposed to [M][N], with the sample indices as values
// (32 x 32 tiles turned in shared memory: both sides are read and written along rows)
__global__ void __launch_bounds__(256) ic_keys_kernel(int64_t N, int M, const float* __restrict__ Rs,
                                                      uint32_t* __restrict__ keys, uint32_t* __restrict__ vals)
{
    __shared__ uint32_t t[32][33];
    const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
    const int64_t k0 = (int64_t)blockIdx.x * 32;
    const int i0 = blockIdx.y * 32;
#pragma unroll
    for (int y = ty; y < 32; y += 8)
        if (k0 + y < N && i0 + tx < M) {
            const uint32_t b = __float_as_uint(Rs[(k0 + y) * M + i0 + tx]);
            t[y][tx] = (b & 0x80000000u) ? ~b : (b | 0x80000000u);
        }
    __syncthreads();
#pragma unroll
    for (int y = ty; y < 32; y += 8)
        if (i0 + y < M && k0 + tx < N) {
            const int64_t o = (int64_t)(i0 + y) * N + k0 + tx;
            keys[o] = t[tx][y];
            vals[o] = (uint32_t)(k0 + tx);
        }
}

// strata [M][N]: sample sorted[i][r] takes stratum r of dimension i
__global__ void ic_ranks_kernel(int64_t N, int M, const uint32_t* __restrict__ sorted, uint32_t* __restrict__ strata)
{
    const int64_t total = N * M;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(t / N);
        const int64_t r = t - (int64_t)i * N;
        strata[(int64_t)i * N + sorted[t]] = (uint32_t)r;
    }
}

__global__ void ic_segments_kernel(int M, int64_t N, int* __restrict__ off)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i <= M) off[i] = (int)((int64_t)i * N);
}

static int ic_grid(int64_t total, int block, int sms)
{
    int64_t g = (total + block - 1) / block;
    const int64_t cap = (int64_t)sms * 32;
    return (int)(g < 1 ? 1 : (g > cap ? cap : g));
}

size_t ic_sort_bytes(int64_t N, int M)
{
    size_t bytes = 0;
    cub::DeviceSegmentedRadixSort::SortPairs(nullptr, bytes, (const uint32_t*)nullptr, (uint32_t*)nullptr,
                                             (const uint32_t*)nullptr, (uint32_t*)nullptr, (int64_t)N * M, M,
                                             (const int*)nullptr, (const int*)nullptr);
    return bytes;
}

cudaError_t launch_ic_strata(uint64_t seed, int64_t N, int M, const IcWork& w, uint32_t* strata, int sms,
                             cudaStream_t st)
{
    if (M > IC_MAX_M || N < 2 || N > 2147483647LL || (int64_t)N * M > 2147483647LL) return cudaErrorInvalidValue;
    const int64_t NM = N * (int64_t)M;
    cudaError_t e;
    ic_score_table_kernel<<<ic_grid(N, 256, sms), 256, 0, st>>>((uint32_t)N, w.a);
    ic_score_moments_kernel<<<1, 1024, 0, st>>>((uint32_t)N, w.a, w.mom);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = launch_design_scores(seed, N, M, w.a, w.mom, w.R, sms, st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(w.G, 0, sizeof(double) * (size_t)M * M, st)) != cudaSuccess) return e;
    const int tiles = (M + IC_GT - 1) / IC_GT;
    const int64_t slices = (N + IC_GRAM_ROWS - 1) / IC_GRAM_ROWS;
    if (slices > 65535) return cudaErrorInvalidValue;
    ic_gram_kernel<<<dim3(tiles, tiles, (unsigned)slices), 256, 0, st>>>(N, M, w.R, w.G);
    ic_corr_kernel<<<(unsigned)(((int64_t)M * M + 255) / 256), 256, 0, st>>>(M, w.G, w.A, w.ok);
    ic_first_block_kernel<<<1, 32, 0, st>>>(M, w.A, w.ok);
    for (int p0 = 0; p0 + IC_NB < M; p0 += IC_NB) {
        const int left = M - p0 - IC_NB;  // rows past the panel's diagonal block
        const unsigned t = (unsigned)((left + 63) / 64);
        ic_panel_kernel<<<(left + 127) / 128, 128, 0, st>>>(M, p0, w.A);
        ic_update_kernel<<<dim3(t, t), 256, 0, st>>>(M, p0, w.A, w.ok);
    }
    // (process-wide attribute, always the same bound: launches may race on it)
    if ((e = cudaFuncSetAttribute(ic_inverse_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  IC_CB * IC_MAX_M * (int)sizeof(float))) != cudaSuccess)
        return e;
    ic_inverse_kernel<<<(M + IC_CB - 1) / IC_CB, 256, IC_CB * M * sizeof(float), st>>>(M, w.A, w.B);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // R* = R Q^-T
    if ((e = launch_sgemm_nn(N, M, M, w.R, w.B, w.Rs, true, st)) != cudaSuccess) return e;
    // keys in place of R, then the sort per column into (Rs, vals_out)
    uint32_t* keys = reinterpret_cast<uint32_t*>(w.R);
    uint32_t* keys_out = reinterpret_cast<uint32_t*>(w.Rs);
    const int64_t kt = (N + 31) / 32;
    ic_keys_kernel<<<dim3((unsigned)kt, (unsigned)((M + 31) / 32)), 256, 0, st>>>(N, M, w.Rs, keys, w.vals);
    ic_segments_kernel<<<(M + 1 + 255) / 256, 256, 0, st>>>(M, N, w.off);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    size_t bytes = w.sort_bytes;
    if ((e = cub::DeviceSegmentedRadixSort::SortPairs(w.sort_tmp, bytes, keys, keys_out, w.vals, w.vals_out, NM, M,
                                                      w.off, w.off + 1, 0, 32, st)) != cudaSuccess)
        return e;
    ic_ranks_kernel<<<ic_grid(NM, 256, sms), 256, 0, st>>>(N, M, w.vals_out, strata);
    return cudaGetLastError();
}

}  // namespace fmc
