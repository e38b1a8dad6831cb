// K dithers per coordinate: counts of non-negative dithered values and their bit planes (Def. 3.7, Remark 3.3).
// A warp works on groups of 128 coordinates: lane l holds coordinates 128 G + 32 r + l, r = 0 .. 3, whose
// four generator outputs of dither k are one call (domain 1 + k, counter 32 G + l).  The dithers of a group can be
// shared among warps: counts are packed four bytes to a word and simply add up (K <= 255).
#pragma once
#include "common.cuh"

namespace fosgd {

// z_k = (2 k24 + 1 - 2^24) dc + y with one rounding: is it non-negative?  What is not a number (infinities among the gradient's
// entries, or one itself) counts as its sign bit says, +, in the tile kernels, and as - in the kernel of short transforms.
template <bool NAN_COUNTS>
__device__ __forceinline__ bool dithered_nonneg(uint32_t k24, float dc, float y)
{
    const float z = fmaf(fmaf((float)k24, 2.f, -16777215.f), dc, y);
    return NAN_COUNTS ? (int)__float_as_uint(z) >= 0 : z >= 0.f;
}

// Smallest k24 in [0, 2^24] (2^24: none) whose dithered value is non-negative.  The value grows with k24, so that
// one comparison of the generator's word replaces conversion, scaling and addition in every further dither:
// a guess by division, good to a few units, is moved until the predicate itself confirms it.
template <bool NAN_COUNTS>
__device__ __forceinline__ uint32_t dither_threshold(float dc, float y)
{
    const float guess = fminf(fmaxf(fmaf(__fdividef(-y, dc), 0.5f, 8388607.5f), 0.f), 16777216.f);   // (NaN -> 0)
    uint32_t k = (uint32_t)guess;
    int steps = 0;
    while (steps < 8 && k > 0u && dithered_nonneg<NAN_COUNTS>(k - 1u, dc, y)) { --k; ++steps; }
    while (steps < 8 && k < 16777216u && !dithered_nonneg<NAN_COUNTS>(k, dc, y)) { ++k; ++steps; }
    if (steps == 8) {   // the guess was far off (dc or y at the ends of the exponent range): bisect
        uint32_t lo = 0u, hi = 16777216u;
        while (lo < hi) {
            const uint32_t mid = (lo + hi) >> 1;
            if (dithered_nonneg<NAN_COUNTS>(mid, dc, y)) hi = mid; else lo = mid + 1u;
        }
        k = lo;
    }
    return k;
}

// From this many dithers on the thresholds (about 20 instructions per coordinate) pay: a dither then costs a compare and
// an add beside its share of the generator call, against five instructions.
constexpr int kThresholdDithers = 8;

// counts over dithers k0 .. k1 - 1 of this lane's four coordinates, one per byte
template <bool NAN_COUNTS>
__device__ __forceinline__ uint32_t dither_counts(const PassParamsRK& p, uint32_t id, uint32_t counter, const float (&y)[4],
                                                  float dc, int k0, int k1)
{
    uint32_t c = 0;
    if (p.K >= kThresholdDithers) {
        uint32_t least[4], one[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const uint32_t k = dither_threshold<NAN_COUNTS>(dc, y[r]);
            least[r] = k << 8;                                  // word >> 8 >= k  <=>  word >= k << 8
            one[r] = k < 16777216u ? 1u << (8 * r) : 0u;
        }
#pragma unroll 2
        for (int k = k0; k < k1; ++k) {
            const uint4 w = rng_words_dither(p, id, 1u + (uint32_t)k, counter);
            if (w.x >= least[0]) c += one[0];
            if (w.y >= least[1]) c += one[1];
            if (w.z >= least[2]) c += one[2];
            if (w.w >= least[3]) c += one[3];
        }
    } else {
#pragma unroll 3
        for (int k = k0; k < k1; ++k) {
            const uint4 w = rng_words_dither(p, id, 1u + (uint32_t)k, counter);
            if (dithered_nonneg<NAN_COUNTS>(w.x >> 8, dc, y[0])) c += 1u;
            if (dithered_nonneg<NAN_COUNTS>(w.y >> 8, dc, y[1])) c += 1u << 8;
            if (dithered_nonneg<NAN_COUNTS>(w.z >> 8, dc, y[2])) c += 1u << 16;
            if (dithered_nonneg<NAN_COUNTS>(w.w >> 8, dc, y[3])) c += 1u << 24;
        }
    }
    return c;
}

// The bit planes of a group's counts: word r of the group (r_first <= r < r_first + nr) of plane b goes to
// dst[b * plane_words + r - r_first].  A whole warp calls it.
__device__ __forceinline__ void store_count_planes(uint32_t counts, uint32_t lane, int P, uint32_t* dst, int64_t plane_words,
                                                   int r_first = 0, int nr = 4)
{
    uint32_t mine = 0;   // lane 4 b + r: word r of plane b
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        if (b < P) {
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const uint32_t word = __ballot_sync(0xFFFFFFFFu, (counts >> (8 * r + b)) & 1u);
                if (lane == 4u * b + r) mine = word;
            }
        }
    }
    const int b = (int)(lane >> 2), r = (int)(lane & 3u) - r_first;
    if (b < P && r >= 0 && r < nr) dst[(int64_t)b * plane_words + r] = mine;
}

}  // namespace fosgd
