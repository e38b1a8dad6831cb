// Transforms shorter than 2^10 (tiny gradients, or small blocks in blocked mode): one thread
// block per transform, the textbook in-place butterfly sweeps in shared memory.  Every source
// and sink of the library in one kernel.  Such calls are all latency: the butterflies cost about a
// microsecond, and the dithers are shared out over all warps (group of 128 coordinates, range of dithers), so
// that K = 255 on one transform of 2^9 is 16 generator calls deep instead of one thread's 8160.
#include <type_traits>

#include "common.cuh"
#include "dither.cuh"

namespace fosgd {

constexpr int kSmallThreads = 512;   // of the dither sinks (K > 1); 128 otherwise

// PACK: the dither sinks.  The others are compiled without them, with a constant number of threads: many short blocks are bound by
// instructions and by how many of them fit an SM (2^22 coordinates in blocks of 32, decode: 229 us in one kernel, 121 without).
// OVERLAP: launched while the kernel in front drains (grids that are not do not pay for the wait).
template <bool PACK, bool OVERLAP>
__global__ void __launch_bounds__(PACK ? kSmallThreads : 128)
small_kernel(const std::conditional_t<PACK, PassParamsRK, PassParams> p, const int L, const int src, const int sink)
{
    __shared__ float x[512];
    __shared__ float acc[512];
    if constexpr (OVERLAP) pdl_begin();
    const int n = 1 << L;
    const int tid = threadIdx.x, nt = PACK ? (int)blockDim.x : 128;
    const int64_t base = (int64_t)blockIdx.x << L;
    const bool loop_workers = !PACK && sink == SINK_FINAL;
    const int w_begin = loop_workers ? 0 : (int)blockIdx.y;
    const int w_end = loop_workers ? p.nworkers : w_begin + 1;
    for (int e = tid; e < n; e += nt) acc[e] = 0.f;

    for (int wk = w_begin; wk < w_end; ++wk) {
        const uint32_t id = p.id0 + (uint32_t)wk;
        const float amp = amplitude_at(p, wk, base);   // one transform never spans two blocks
        __syncthreads();
        for (int e = tid; e < n; e += nt) {
            const int64_t i = base + e;
            float v;
            if (src == SRC_G32) {
                v = (i < p.d) ? (static_cast<const float*>(p.src) + (int64_t)wk * p.src_stride)[i] : 0.f;
            } else if (src == SRC_G16) {
                const uint16_t* g = static_cast<const uint16_t*>(p.src) + (int64_t)wk * p.src_stride;
                v = (i < p.d) ? __uint_as_float((uint32_t)g[i] << 16) : 0.f;
            } else if (src == SRC_WS) {
                v = (static_cast<const float*>(p.src) + (int64_t)wk * p.src_stride)[i];
            } else {
                const uint32_t* b = static_cast<const uint32_t*>(p.src) + (int64_t)wk * p.src_stride + (i >> 5);
                v = plane_value(b, p.dp >> 5, p.P, p.K, (uint32_t)i & 31u);
            }
            if (src == SRC_G32 || src == SRC_G16)
                v = flip_by_bit(v, eps_word(p.rng, id, (uint32_t)(i >> 5)), (uint32_t)i & 31u);
            x[e] = v;
        }
        __syncthreads();
        for (int h = 1; h < n; h <<= 1) {
            for (int j = tid; j < n / 2; j += nt) {
                const int idx = ((j & ~(h - 1)) << 1) | (j & (h - 1));
                const float a = x[idx], b = x[idx + h];
                x[idx] = a + b;
                x[idx + h] = a - b;
            }
            __syncthreads();
        }
        if constexpr (PACK) {
            // groups of 128 coordinates: four words, or the n / 32 words of a shorter transform inside its group
            __shared__ uint32_t counts[4 * 32];
            const int warp = tid >> 5, lane = tid & 31, warps = nt / 32;
            const int ngroups = n >= 128 ? n / 128 : 1, nr = n >= 128 ? 4 : n / 32, r_first = (int)(base >> 5) & 3;
            const int share = warps / ngroups;                    // (both powers of two, warps >= 4)
            const int g = warp / share, k0 = p.K * (warp % share) / share, k1 = p.K * (warp % share + 1) / share;
            if (tid < 128) counts[tid] = 0u;
            __syncthreads();
            float y[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int word = 4 * g + r - (n >= 128 ? 0 : r_first);
                y[r] = word >= 0 && word < n / 32 ? x[32 * word + lane] : 0.f;
            }
            const uint32_t c = dither_counts<false>(p, id, (((uint32_t)(base >> 7) + (uint32_t)g) << 5) + (uint32_t)lane, y,
                                             p.dither_c * amp, k0, k1);
            atomicAdd(counts + 32 * g + lane, c);
            __syncthreads();
            uint32_t* dst = static_cast<uint32_t*>(p.dst) + (int64_t)wk * p.dst_stride + (base >> 5);
            if (warp < ngroups)
                store_count_planes(counts[32 * warp + lane], (uint32_t)lane, p.P, dst + 4 * warp, p.dp >> 5, n >= 128 ? 0 : r_first, nr);
        } else if (sink == SINK_WS) {
            float* dst = static_cast<float*>(p.dst) + (int64_t)wk * p.dst_stride;
            for (int e = tid; e < n; e += nt) dst[base + e] = x[e] * p.scale;
        } else {
            for (int e = tid; e < n; e += nt) {
                const int64_t i = base + e;
                const float f = flip_by_bit(x[e], eps_word(p.rng, id, (uint32_t)(i >> 5)), (uint32_t)i & 31u);
                acc[e] = fmaf(f, p.amp_mode == AMP_WEIGHT ? amp : 1.f, acc[e]);
            }
        }
    }
    if (loop_workers) {
        float* dst = static_cast<float*>(p.dst);
        const float sc = p.scale * (p.amp_mode == AMP_SCALE ? amplitude_at(p, 0, base) : 1.f);
        for (int e = tid; e < n; e += nt) {
            const int64_t i = base + e;
            if (i < p.d_out) {
                store_final(dst + i, acc[e], sc, p.overwrite);
            }
        }
    }
}

cudaError_t launch_small(int L, int src, int sink, const PassParams& p, cudaStream_t s)
{
    if (L < 5 || L > 9) return cudaErrorInvalidValue;
    const dim3 grid((unsigned)(p.dp >> L), sink == SINK_FINAL ? 1u : (unsigned)p.nworkers);
    const unsigned threads = sink == SINK_PACKK ? kSmallThreads : 128;
    // blocks that walk several workers last: where the grid is neither small nor full, those that start early crowd on the
    // SMs that have room (2^17 coordinates in blocks of 2^8, eight workers: 28 us overlapped, 21 not)
    const int64_t limit = sink == SINK_FINAL && p.nworkers > 1 ? 1 << 14 : kOverlapThreads;
    if (sink == SINK_PACK1 || sink == SINK_PACKK)
        return launch_either<small_kernel<true, true>, small_kernel<true, false>>(grid, threads, s, limit, with_round_keys(p), L, src, sink);
    return launch_either<small_kernel<false, true>, small_kernel<false, false>>(grid, threads, s, limit, p, L, src, sink);
}

}  // namespace fosgd
