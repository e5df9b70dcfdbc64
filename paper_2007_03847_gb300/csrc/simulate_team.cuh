// Algorithm 1 steps 2-4 fused for few samples (up to 16 machines): one CTA per 32
// samples, the machines of a sample spread over a team of L warps.
//
// What bounds a small study is the latency of one sample's step: with one thread per
// sample a step of ten machines is 6400 cycles of one warp's dependent instructions
// while most of the GPU idles.  Here lane = sample and warp i of the team integrates
// machine i, so that a stage is some 90 instructions per warp and two or three warps
// share a scheduler and fill each other's waits; 32 samples take a CTA (and, while
// there are SMs, an SM), and everything that is not the step itself is taken out of the
// team's warps:
//
//   warp 0      issues TMA and tcgen05.mma of the next chunk's increments and turns
//               them into the disturbances' paths (Euler-Maruyama, the smooth form's
//               stage values, or the per-step normals), double-buffered in shared memory
//   warp 1      forms every step's moment triples (column_sums) and the response
//               function from a double-buffered ring of states
//   warps 2 ..  the team: per RK stage each publishes its machine's (cos - 1, sin) and
//               meets the others at one named barrier; its row of the network stays in
//               registers (packed FP32 with a constant-bank operand costs a lone warp 5
//               cycles, with registers 2.3)
//
// The FP32 operations and their order per value are those of simulate_fused_kernel:
// the network sums run over j in ascending order (a machine's own column and the
// padding are zero terms), the angle tier is that of the 32 samples and all their
// machines (the barrier carries whether all warps are in the shortest series' range;
// otherwise they exchange their tiers, and the rare stage whose tier differs from the
// one before redoes its sines), so both kernels give the same bits.  The triples leave per
// group of 32 samples ([group][Nt+1][ref | dev | m2]); the reduction combines four into a
// tile's as the per-sample kernel's flush does.
// Measured (GB300): see team_fits in api.cu.
#pragma once

#include "fmc_common.cuh"
#include "kernels.cuh"
#include "swing.cuh"
#include "tc_common.cuh"

namespace fmc {

constexpr int TEAM_ROWS = 32;  // samples per CTA
constexpr int TEAM_MB = 4;     // steps per moment buffer

__host__ __device__ constexpr int team_threads(int nm) { return 64 + 32 * nm; }

struct TeamArgs {
    int64_t count;
    int Nt, TC, d, Ks, nkb, split;
    int ns;  // ring stages
    uint32_t tmem_cols;
    float* part;  // [groups][Nt+1][3][2n]
    float* traj;  // [count][Nt+1][2n] or nullptr
    int* err;
    EmSpec em;
    double* rrf;
};

// Shared memory (bytes past the 1 KB alignment): the ring (A tiles of 32 rows; an MMA
// reads 128 rows, so 8 KB follow the last tile), two path buffers, two exchange
// buffers, two moment buffers.
struct TeamSmem {
    int paths, exch, mom, total;
};
__host__ __device__ inline TeamSmem team_smem(int nm, int TC, int d, int split, int ns, bool smooth)
{
    const int stage = (TEAM_ROWS * 64 + (smooth ? 2 : 1) * TC * 64) * (split ? 2 : 1);
    TeamSmem s;
    s.paths = ns * stage + 8192;
    s.exch = s.paths + 2 * TC * d * (smooth ? 4 : 1) * 128;
    s.mom = s.exch + 2 * (nm * 256 + 128 + 16);
    s.total = s.mom + 2 * TEAM_MB * (32 * (2 * nm + 1) + 2 * nm) * 4;
    return s;
}

template <int N>
__device__ __forceinline__ void team_bar()
{
    if constexpr (N > 1) asm volatile("bar.sync 1, %0;" ::"n"(N * 32) : "memory");
}

// Whether p holds in every thread of the team.
template <int N>
__device__ __forceinline__ bool team_all(bool p)
{
    if constexpr (N == 1) return __all_sync(0xffffffffu, p);
    int r;
    asm volatile(
        "{\n\t.reg .pred q, o;\n\tsetp.ne.s32 q, %1, 0;\n\t"
        "bar.red.and.pred o, 1, %2, q;\n\tselp.s32 %0, 1, 0, o;\n\t}"
        : "=r"(r)
        : "r"((int)p), "n"(N * 32)
        : "memory");
    return r != 0;
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Bounded wait that polls before it sleeps (the producers are normally ahead).
__device__ __forceinline__ bool team_wait(uint64_t* bar, uint32_t parity)
{
    for (int it = 0; it < 64; ++it)
        if (mbar_try_wait(bar, parity)) return true;
    return mbar_wait(bar, parity);
}

// (cos - 1, sin) of a deviation by the series of the (warp-uniform) tier.
__device__ __forceinline__ float2 team_trig(int tier, float a)
{
    float2 r;
    if (tier == 0)
        deviation_trig1<0>(a, &r.y, &r.x);
    else if (tier == 1)
        deviation_trig1<1>(a, &r.y, &r.x);
    else if (tier == 2)
        deviation_trig1<2>(a, &r.y, &r.x);
    else
        deviation_trig1<3>(a, &r.y, &r.x);
    return r;
}

template <int NM, int ND, bool SMOOTH>
__global__ void __launch_bounds__(team_threads(NM), NM > 8 ? 1 : 2)
    simulate_team_kernel(const __grid_constant__ SwingParams<NM, ND> p, const __grid_constant__ CUtensorMap mAh,
                         const __grid_constant__ CUtensorMap mAl, const __grid_constant__ CUtensorMap mBh,
                         const __grid_constant__ CUtensorMap mBl, const TeamArgs a)
{
    constexpr bool SHORT = !SMOOTH && NM <= 10;  // the tiers simulate_fused_kernel's step takes
    constexpr int TIER0 = SHORT ? 0 : 2;
    constexpr int WROW = 2 * NM + 1;
    constexpr int SST = 32 * WROW + 2 * NM;  // floats per step of a moment buffer (lanes of two steps on different banks)
    constexpr int XV = SMOOTH ? 4 : 1;       // path values per step and disturbance
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    __shared__ uint64_t bars[2 * TC_MAX_STAGES + 1];                // full[ns], freed[ns], done
    __shared__ uint64_t xfull[2], xfree[2], mfull[2], mfree[2];     // path and moment buffers
    __shared__ uint32_t tmem_base;

    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const int n = p.n, d = p.d, S = 2 * n, S3 = 3 * S;
    const int64_t row0 = (int64_t)blockIdx.x * TEAM_ROWS;
    const int64_t srow = row0 + lane;
    const bool active = srow < a.count;
    const int na = a.count - row0 >= 32 ? 32 : (int)(a.count - row0);
    const int TC = a.TC, CW = SMOOTH ? 2 * TC : TC;
    const TeamSmem lay = team_smem(NM, TC, d, a.split, a.ns, SMOOTH);
    float* paths = reinterpret_cast<float*>(smem + lay.paths);  // [2][TC][d][XV][32]
    const int xbuf = TC * d * XV * 32;
    // per exchange buffer: (cos - 1, sin) [NM][32], machine 0's speed [32], the warps' tiers (bytes [16])
    uint8_t* exch = smem + lay.exch;
    constexpr int EXCH = NM * 256 + 128 + 16;  // (see team_smem)
    float* mom = reinterpret_cast<float*>(smem + lay.mom);  // [2][TEAM_MB][SST]
    const bool em = a.em.on != 0;

    if (tid == 0) {
        if (!em) {
            prefetch_tmap(&mAh);
            prefetch_tmap(&mBh);
        }
        for (int b = 0; b < 2 * TC_MAX_STAGES + 1; ++b) mbar_init(&bars[b], 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&xfull[b], 1);
            mbar_init(&xfree[b], NM);
            mbar_init(&mfull[b], NM);
            mbar_init(&mfree[b], 1);
        }
        fence_mbar_init();
    }
    if (warp == 0) tmem_alloc(&tmem_base, a.tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;

    if (warp == 0) {
        // ---- increments and disturbance paths, a chunk ahead of the team ----
        TcRing r;
        r.a_bytes = TEAM_ROWS * 64;
        r.b_bytes = CW * 64;
        r.split = a.split;
        r.base = smem;
        r.ns = (uint32_t)a.ns;
        r.full = &bars[0];
        r.freed = &bars[TC_MAX_STAGES];
        uint64_t* done = &bars[2 * TC_MAX_STAGES];
        const int J = d * a.nkb;
        const uint32_t idesc = umma_idesc_bf16(TC_M, CW);
        uint32_t g = 0;
        float x[ND], f0[ND];
#pragma unroll
        for (int q = 0; q < ND; ++q) {
            x[q] = 0.f;
            f0[q] = 0.f;
        }
        uint32_t nm = 0;  // contractions so far
        int c = 0;        // path buffers so far
        for (int n0 = SMOOTH ? -TC : 0; n0 < a.Nt; n0 += TC) {
            if (!em) {
                int ok = 1;
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    tc_fence_after();
                    auto load_item = [&](int j) {
                        const int wj = j / a.nkb, kb = j - wj * a.nkb;
                        return ring_load(r, g + (uint32_t)j, &mAh, &mAl, &mBh, &mBl, wj * a.Ks + kb * TC_BK, (int)row0,
                                         kb * TC_BK, SMOOTH ? 2 * n0 + 1 : n0);
                    };
                    bool good = true;
                    int issued = 0;
                    for (; issued < J && issued + 1 < (int)r.ns && good; ++issued) good = load_item(issued);
                    for (int j = 0; j < J && good; ++j) {
                        if (issued < J) {
                            good = load_item(issued);
                            ++issued;
                            if (!good) break;
                        }
                        const int wj = j / a.nkb, kb = j - wj * a.nkb;
                        good = ring_mma(r, g + (uint32_t)j, tmem + (uint32_t)(wj * CW), idesc, kb == 0);
                    }
                    g += (uint32_t)J;
                    if (good)
                        umma_commit(done);
                    else
                        atomicExch(a.err, DEV_TIMEOUT_TMA);
                    ok = good ? 1 : 0;
                }
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) break;
                ok = mbar_wait(done, nm & 1u) ? 1 : 0;
                ++nm;
                if (!__all_sync(0xffffffffu, ok)) {
                    atomicExch(a.err, DEV_TIMEOUT_MMA);
                    break;
                }
                tc_fence_after();
                if constexpr (SMOOTH) {
                    if (n0 < 0) {
                        // f(0): the last column of the contraction over the rows up to 0
#pragma unroll
                        for (int q = 0; q < ND; ++q)
                            if (q < d) f0[q] = tmem_ld1(tmem + (uint32_t)(q * CW + CW - 1));
                        tmem_ld_wait();
                        continue;
                    }
                }
            }
            const int b = c & 1;
            if (c >= 2) {
                const int ok = team_wait(&xfree[b], (uint32_t)((c >> 1) - 1) & 1u) ? 1 : 0;
                if (!__all_sync(0xffffffffu, ok)) {
                    atomicExch(a.err, DEV_TIMEOUT_MMA);
                    break;
                }
            }
            float* xb = paths + b * xbuf + lane;
            const int steps = (a.Nt - n0) < TC ? (a.Nt - n0) : TC;
            if constexpr (SMOOTH) {
#pragma unroll 1
                for (int s = 0; s < steps; ++s) {
                    float fh[ND], f1[ND], xst[4][ND];
#pragma unroll
                    for (int q = 0; q < ND; ++q) {
                        fh[q] = 0.f;
                        f1[q] = 0.f;
                    }
#pragma unroll
                    for (int q = 0; q < ND; ++q)
                        if (q < d) {
                            fh[q] = tmem_ld1(tmem + (uint32_t)(q * CW + 2 * s));
                            f1[q] = tmem_ld1(tmem + (uint32_t)(q * CW + 2 * s + 1));
                        }
                    tmem_ld_wait();
                    smooth_stages<NM, ND>(p, n0 + s, x, f0, fh, f1, xst);
#pragma unroll
                    for (int q = 0; q < ND; ++q) {
                        f0[q] = f1[q];
                        if (q < d) {
                            float* o = xb + (s * d + q) * (4 * 32);
                            o[0] = xst[1][q];
                            o[32] = xst[2][q];
                            o[64] = xst[3][q];
                            o[96] = x[q];
                        }
                    }
                }
            } else {
#pragma unroll
                for (int q = 0; q < ND; ++q) {
                    if (q >= d) continue;
                    const float oa = p.ou_a[q], os = p.ou_s[q];
                    float xq = x[q];
#pragma unroll 1
                    for (int s0 = 0; s0 < steps; s0 += 8) {
                        float v[8];
                        if (em) {
#pragma unroll 1
                            for (int j = 0; j < 8; ++j) {
                                const float e = a.em.sqdt * em_normal((uint32_t)(a.em.k0 + srow), q, n0 + s0 + j,
                                                                      a.em.key0, a.em.key1);
                                xq = p.ito.on ? ito_step1<ND>(p.ito, q, oa, os, xq, e, p.dt) : fmaf(oa, xq, os * e);
                                xb[((s0 + j) * d + q) * 32] = xq;
                            }
                            continue;
                        }
                        tmem_ld8(tmem + (uint32_t)(q * TC + s0), v);
                        tmem_ld_wait();
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            xq = p.ito.on ? ito_step1<ND>(p.ito, q, oa, os, xq, v[j], p.dt) : fmaf(oa, xq, os * v[j]);
                            xb[((s0 + j) * d + q) * 32] = xq;
                        }
                    }
                    x[q] = xq;
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&xfull[b]);
            ++c;
        }
    } else if (warp == 1) {
        // ---- moments and the response function ----
        float* out = a.part + (int64_t)blockIdx.x * (a.Nt + 1) * S3;
        // time 0: every sample sits at the (rounded) shift
        for (int v = lane; v < S3; v += 32) out[v] = 0.f;
        float racc = 0.f;  // sum over the grid of the squared centre-of-inertia speed
        for (int m = 0; m * TEAM_MB < a.Nt; ++m) {
            const int b = m & 1;
            const int ok = team_wait(&mfull[b], (uint32_t)(m >> 1) & 1u) ? 1 : 0;
            if (!__all_sync(0xffffffffu, ok)) {
                atomicExch(a.err, DEV_TIMEOUT_MMA);
                break;
            }
            const float* mb = mom + b * TEAM_MB * SST;
            const int t0 = m * TEAM_MB;
            const int nst = a.Nt - t0 < TEAM_MB ? a.Nt - t0 : TEAM_MB;
            for (int e = lane; e < nst * S; e += 32) {
                const int sl = e / S, j = e - sl * S;
                float rf, dv, m2;
                column_sums(mb + sl * SST + (j < n ? j : NM + j - n), WROW, na, &rf, &dv, &m2);
                float* o = out + (int64_t)(t0 + sl + 1) * S3;
                o[j] = rf;
                o[S + j] = dv;
                o[2 * S + j] = m2;
            }
            if (a.rrf)
                for (int sl = 0; sl < nst; ++sl) {
                    const float* row = mb + sl * SST + lane * WROW + NM;
                    float cs = 0.f;
#pragma unroll
                    for (int i = 0; i < NM; ++i) cs = fmaf(p.hw[i], row[i], cs);
                    racc = fmaf(cs, cs, racc);
                }
            __syncwarp();
            if (lane == 0) mbar_arrive(&mfree[b]);
        }
        if (a.rrf) rrf_accumulate(active ? sqrtf(racc / (float)a.Nt) : 0.f, a.rrf);
    } else {
        // ---- the team: warp i integrates machine i ----
        const int i = warp - 2;
        // this machine's row of the network (packed halves, zero on the diagonal) and constants
        unsigned long long P1[NM], P2[NM];
#pragma unroll
        for (int j = 0; j < NM; ++j) {
            P1[j] = *reinterpret_cast<const unsigned long long*>(&p.P1[i][j]);
            P2[j] = *reinterpret_cast<const unsigned long long*>(&p.P2[i][j]);
        }
        const float pst = p.pst[i], qst = p.qst[i], Dh = p.Dh[i], dst = p.dst[i];
        float inj[ND];
#pragma unroll
        for (int q = 0; q < ND; ++q) inj[q] = p.injh[i][q];
        float del = 0.f, w = 0.f, theta = 0.f, x0[ND];
#pragma unroll
        for (int q = 0; q < ND; ++q) x0[q] = 0.f;
        const int64_t trow = 2 * (int64_t)n;
        float* traj = (a.traj != nullptr && active && i < n) ? a.traj + srow * (int64_t)(a.Nt + 1) * trow : nullptr;
        if (traj) {
            traj[i] = dst;
            traj[n + i] = 0.f;
        }
        const float dt = p.dt;
        const bool rk4 = (p.integrator == FMC_RK4);
        const float dth = 0.5f * dt, dtw = dt * p.omega_s, dthw = dth * p.omega_s;
        const float ref = p.rel ? 1.f : 0.f;
        const float hh = rk4 ? dt * (1.0f / 6.0f) : 0.5f * dt;
        const float hhw = hh * p.omega_s;
        int tier = TIER0;  // of the stage before
        int gb = 0;        // exchange buffer
        bool bad = false;
        for (int c = 0, n0 = 0; n0 < a.Nt; ++c, n0 += TC) {
            const int xbi = c & 1;
            if (!bad && !team_wait(&xfull[xbi], (uint32_t)(c >> 1) & 1u)) {
                bad = true;
                atomicExch(a.err, DEV_TIMEOUT_MMA);
            }
            if (!team_all<NM>(!bad)) break;
            const float* xb = paths + xbi * xbuf + lane;
            const int steps = (a.Nt - n0) < TC ? (a.Nt - n0) : TC;
#pragma unroll 1
            for (int s = 0; s < steps; ++s) {
                const int t = n0 + s;
                const int mi = t / TEAM_MB, ms = t % TEAM_MB;
                if (ms == 0 && mi >= 2 && !bad && !team_wait(&mfree[mi & 1], (uint32_t)((mi >> 1) - 1) & 1u)) {
                    bad = true;
                    atomicExch(a.err, DEV_TIMEOUT_MMA);
                }
                // the disturbances at t_n and t_{n+1} (the smooth form: their stage values)
                float x1[ND], xst[SMOOTH ? 4 : 1][ND];
                const float ev = t >= p.ev_step ? 1.f : 0.f;
#pragma unroll
                for (int q = 0; q < ND; ++q) {
                    x1[q] = 0.f;
                    if constexpr (SMOOTH) {
                        const float e = q == p.ev_slot ? ev : 0.f;
                        xst[0][q] = q < d ? x0[q] : e;
                        const float* o = xb + (s * d + q) * (4 * 32);
                        xst[1][q] = q < d ? o[0] : e;
                        xst[2][q] = q < d ? o[32] : e;
                        xst[3][q] = q < d ? o[64] : e;
                        x1[q] = q < d ? o[96] : e;
                    } else {
                        if (q < d) x1[q] = xb[(s * d + q) * 32];
                        if (q == p.ev_slot) {
                            x0[q] = ev;
                            x1[q] = ev;
                        }
                    }
                }
                // the forcing at the stage times (the two middle stages share theirs)
                float f0 = 0.f, fm = 0.f, fm2 = 0.f, f1 = 0.f;
#pragma unroll
                for (int q = 0; q < ND; ++q) {
                    if constexpr (SMOOTH) {
                        f0 = fmaf(inj[q], xst[0][q], f0);
                        fm = fmaf(inj[q], xst[1][q], fm);
                        fm2 = fmaf(inj[q], xst[2][q], fm2);
                        f1 = fmaf(inj[q], xst[3][q], f1);
                    } else {
                        const float dx = x1[q] - x0[q];
                        f0 = fmaf(inj[q], fmaf(0.f, dx, x0[q]), f0);
                        fm = fmaf(inj[q], fmaf(0.5f, dx, x0[q]), fm);
                        f1 = fmaf(inj[q], fmaf(1.f, dx, x0[q]), f1);
                    }
                }
                if (!SMOOTH) fm2 = fm;
                float ad = 0.f, aw = 0.f, yd = del, yw = w, ath = 0.f;
                auto stage = [&](float b, float cn, float cnw, float f) {
                    // publish the stage input's sines (at the last stage's tier) and machine
                    // 0's speed
                    float2* cs = reinterpret_cast<float2*>(exch + gb * EXCH);
                    float* w0s = reinterpret_cast<float*>(exch + gb * EXCH + NM * 256);
                    uint8_t* tiers = exch + gb * EXCH + NM * 256 + 128;
                    gb ^= 1;
                    float2 my;
                    if (tier == TIER0)
                        deviation_trig1<TIER0>(yd, &my.y, &my.x);
                    else
                        my = team_trig(tier, yd);
                    float w0 = yw * ref;
                    if constexpr (NM > 1) {
                        cs[i * 32 + lane] = my;
                        if (i == 0) w0s[lane] = w0;
                    }
                    const uint32_t mx = __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(0.f, fabsf(yd))));
                    bool ask = tier != TIER0;
                    if (!ask) ask = !team_all<NM>(mx <= __float_as_uint(SHORT ? 0.05f : 0.8f));
                    if (ask) {
                        // some warp is past the shortest series (or the last stage was)
                        int now = mx <= __float_as_uint(0.8f) ? 2 : 3;
                        if (SHORT) now = mx <= __float_as_uint(0.05f) ? 0 : (mx <= __float_as_uint(0.25f) ? 1 : now);
                        if constexpr (NM > 1) {
                            if (lane == 0) tiers[i] = (uint8_t)now;
                            team_bar<NM>();
#pragma unroll 1
                            for (int j = 0; j < NM; ++j) now = max(now, (int)tiers[j]);
                        }
                        if (now != tier) {
                            // (uniform over the team) another tier: the sines again
                            tier = now;
                            my = team_trig(tier, yd);
                            if constexpr (NM > 1) {
                                cs[i * 32 + lane] = my;
                                team_bar<NM>();
                            }
                        }
                    }
                    if constexpr (NM > 1) w0 = w0s[lane];
                    ath = fmaf(b, w0, ath);
                    // network sums (row_network)
                    unsigned long long au = 0ull, av = 0ull;
                    if constexpr (NM > 1) {
#pragma unroll
                        for (int j = 0; j < NM; ++j) {
                            const unsigned long long c2 = *reinterpret_cast<const unsigned long long*>(&cs[j * 32 + lane]);
                            au = ffma2(P1[j], c2, au);
                            av = ffma2(P2[j], c2, av);
                        }
                    }
                    float u0, u1, v0, v1;
                    f2unpack(au, u0, u1);
                    f2unpack(av, v0, v1);
                    const float U = u0 + u1;
                    float V = v0 + v1;
                    V += qst;
                    float dpe = fmaf(my.x, U + pst, U);
                    dpe = fmaf(my.y, V, dpe);
                    const float kw = fmaf(-Dh, yw, f - dpe);
                    const float kv = yw - w0;
                    ad = fmaf(b, kv, ad);
                    aw = fmaf(b, kw, aw);
                    yd = fmaf(cnw, kv, del);
                    yw = fmaf(cn, kw, w);
                };
                if (rk4) {
                    stage(1.f, dth, dthw, f0);
                    stage(2.f, dth, dthw, fm);
                    stage(2.f, dt, dtw, fm2);
                    stage(1.f, dth, dthw, f1);
                } else {
                    stage(1.f, dt, dtw, f0);
                    stage(1.f, dt, dtw, SMOOTH ? fm : f1);
                }
                del = fmaf(hhw, ad, del);
                w = fmaf(hh, aw, w);
                theta = fmaf(hhw, ath, theta);
#pragma unroll
                for (int q = 0; q < ND; ++q) x0[q] = x1[q];
                if (traj) {
                    float* o = traj + (int64_t)(t + 1) * trow;
                    o[i] = (theta + del) + dst;
                    o[n + i] = w;
                }
                float* row = mom + ((mi & 1) * TEAM_MB + ms) * SST + lane * WROW;
                row[i] = theta + del;
                row[NM + i] = w;
                if (ms == TEAM_MB - 1 || t == a.Nt - 1) {
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&mfull[mi & 1]);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&xfree[xbi]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, a.tmem_cols);
}

template <int NM, int ND>
cudaError_t launch_team_t(const void* params, const CUtensorMap* maps, const TeamArgs& a, int smooth, cudaStream_t st,
                          int* max_ctas_per_sm)
{
    const SwingParams<NM, ND>& p = *static_cast<const SwingParams<NM, ND>*>(params);
    auto kern = smooth ? simulate_team_kernel<NM, ND, true> : simulate_team_kernel<NM, ND, false>;
    // (process-wide attribute, always the same bound: launches may race on it)
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM_DYN_MAX);
    if (e != cudaSuccess) return e;
    int smem = 1024 + team_smem(NM, a.TC, a.d, a.split, a.ns, smooth != 0).total;
    // no more CTAs on an SM than its 512 TMEM columns hold
    const int floor = 233472 / (512 / (int)a.tmem_cols + 1) - 1024 + 64;
    if (smem < floor) smem = floor;
    if (smem > TC_SMEM_DYN_MAX) return cudaErrorInvalidValue;
    if (max_ctas_per_sm) {
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(max_ctas_per_sm, kern, team_threads(NM), smem);
        if (e != cudaSuccess) return e;
    }
    const int64_t groups = (a.count + TEAM_ROWS - 1) / TEAM_ROWS;
    kern<<<(unsigned)groups, team_threads(NM), smem, st>>>(p, maps[0], maps[1], maps[2], maps[3], a);
    return cudaGetLastError();
}

}  // namespace fmc
