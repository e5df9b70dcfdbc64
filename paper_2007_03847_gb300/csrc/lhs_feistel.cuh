// The per-dimension stratum permutation of the Latin hypercube design
// (Section IV-B step 1): a keyed balanced Feistel network with cycle walking,
// stateless, so that any (sample, dimension) is computed on its own.
#pragma once

#include <stdint.h>

#include "fmc_common.cuh"

namespace fmc {

constexpr int kFeistelRounds = 6;

// Balanced Feistel network on 2h bits: six rounds (L, R) -> (R, L ^ f_r(R)) with
// f_r(R) = Philox word 0 of the counter (R, dim, 1 + r, 0), masked to h bits;
// pi_dim(k) is the first iterate of it from k that falls in [0, N) (cycle walking
// ends: the cycle through k < N returns to [0, N) within 4^h - N + 1 applications).
// walk: N < 4^h, some values fall outside (every N that is no power of four, also above
// 2^30, where h = 16 and 4^h no longer fits 32 bits; the correlation-reducing
// permutation of one column takes N up to 2^31 - 1).
struct FeistelShape {
    int h;
    uint32_t mask;
    bool walk;
};

inline FeistelShape feistel_shape(int64_t N)
{
    int b = 0;
    while ((int64_t(1) << b) < N) ++b;
    int h = (b + 1) / 2;
    if (h < 1) h = 1;
    FeistelShape f;
    f.h = h;
    f.mask = (h >= 32) ? 0xFFFFFFFFu : ((1u << h) - 1u);
    f.walk = ((uint64_t)1 << (2 * h)) > (uint64_t)N;
    return f;
}

}  // namespace fmc
