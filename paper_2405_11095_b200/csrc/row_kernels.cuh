// Contiguous-tile pass: all T = log2(tile) butterfly stages of the index bits [0, T) on tiles of
// 2^T consecutive coordinates, fused with its source (gradient load + pad + flip, packed bits,
// or an intermediate of an earlier pass) and its sink (dither + sign + pack, fp32 store, or
// flip + sum over workers).  One thread block works on one tile at a time; every thread keeps
// 32 values in registers and the block runs three register rounds of up to five stages each,
// exchanging through shared memory (row pitch 36 words: no bank conflicts in any round).
//
//   round F: register bits 10 .. T-1 and, up to five, the lowest (vector loads) and bits 9, 8, 7
//   round M: register bits 0 .. 4, lane = bits 5 .. 9    (128-bit shared loads and stores)
//   round L: register bits 5 .. 9, lane = bits 0 .. 4, so lane r can own packed word r
//
// A bit that two rounds hold is transformed by the first and rides along in the second.  All bits
// above 9 are done in round F, so from then on a warp works on 1024 consecutive coordinates of its
// own: one block-wide barrier per tile, between F and M, and none between M and L.  (Earlier form:
// F on {0, 1, T-3 .. T-1}, M on {2, 3, 4, 10, 11} with 32-bit accesses and a second block barrier.)
//
// Two kernels share these rounds:
//   row_kernel        source read by the threads themselves: gradients and packed bits (the
//                     single-pass case, transform length <= 2^15), and fp32 intermediates on the way
//                     to a dither sink or with a tile too large for a separate landing buffer.
//   row_stream_kernel source = intermediate of the strided passes, fetched tile by tile with
//                     the bulk async copy engine (cp.async.bulk + mbarrier) into a landing
//                     buffer beside the work tile: the copy of tile k+1 starts as soon as
//                     round F has read tile k, and runs underneath the other rounds and the sink.
#pragma once
#include "common.cuh"
#include "dither.cuh"

namespace fosgd {

__host__ __device__ constexpr int nth_set_bit(uint32_t mask, int n)
{
    for (int b = 0; b < 32; ++b)
        if ((mask >> b) & 1u) {
            if (n == 0) return b;
            --n;
        }
    return -1;
}

// tile offset addressed by register r when the register bits are the set bits of `mask`
__host__ __device__ constexpr int reg_offset(uint32_t mask, int r)
{
    int e = 0;
    for (int rb = 0; rb < 5; ++rb)
        if ((r >> rb) & 1) e |= 1 << nth_set_bit(mask, rb);
    return e;
}

// register-level stage mask: register bit rb is active iff its tile bit is not done yet
__host__ __device__ constexpr int active_mask(uint32_t mask, uint32_t done)
{
    int a = 0;
    for (int rb = 0; rb < 5; ++rb)
        if (!((done >> nth_set_bit(mask, rb)) & 1u)) a |= 1 << rb;
    return a;
}

__host__ __device__ constexpr int phys(int e) { return e + ((e >> 5) << 2); }

// spread the thread index over the tile bits that are not register bits (lowest first)
template <uint32_t MASK, int T>
__device__ __forceinline__ int deposit(int tid)
{
    int e = 0, k = 0;
#pragma unroll
    for (int b = 0; b < T; ++b)
        if (!((MASK >> b) & 1u)) {
            e |= ((tid >> k) & 1) << b;
            ++k;
        }
    return e;
}

template <int T>
struct RowCfg {
    static constexpr int NT = 1 << (T - 5);
    static constexpr int VB = (T >= 15) ? 0 : (T == 14 ? 1 : 2);      // log2 of the vector of a round-F load
    static constexpr uint32_t FMASK = ((1u << VB) - 1u) | (((1u << (5 - VB)) - 1u) << (T - (5 - VB)));
    static constexpr uint32_t MMASK = 0x1Fu;
    static constexpr uint32_t LMASK = 0x3E0u;
    static constexpr int ACT_M = active_mask(MMASK, FMASK);
    static constexpr int ACT_L = active_mask(LMASK, FMASK | MMASK);
    static constexpr int TILE_WORDS = phys(1 << T);
    static constexpr int FLIP_WORDS = (1 << T) / 32;
    static constexpr size_t SMEM_BYTES = (size_t)(TILE_WORDS + FLIP_WORDS) * 4 + 16;  // + mbarrier
    static constexpr size_t EARLY_AT = (SMEM_BYTES + 15) / 16 * 16;                   // the dither words of EARLY
    static constexpr size_t TOP_AT = EARLY_AT;                                        // the planes of SRC_BITS_TOP
    static constexpr size_t TOP_SMEM_BYTES = TOP_AT + (size_t)(kTopStages + 1) * NT * 4;
    static constexpr size_t EARLY_SMEM_BYTES = EARLY_AT + ((size_t)4 << T);
    static_assert(((FMASK | MMASK | LMASK) & ((1u << T) - 1)) == ((1u << T) - 1), "bits uncovered");
};

// parameter block of a kernel by its sink: the dither sinks carry the generator's round keys
template <int SINK> struct KernelParams { using type = PassParams; };
template <> struct KernelParams<SINK_PACK1> { using type = PassParamsRK; };
template <> struct KernelParams<SINK_PACKK> { using type = PassParamsRK; };
template <int SINK>
inline typename KernelParams<SINK>::type kernel_params(const PassParams& p)
{
    if constexpr (SINK == SINK_PACK1 || SINK == SINK_PACKK) return with_round_keys(p);
    else return p;
}

// Registers are capped at 64 per thread (2048 resident threads per SM).  The store and dither
// sinks need no more by themselves.  The flip + accumulate sink holds 32 values and 32 sums per
// thread and would take ~95: capped, it spills a few words but runs twice the warps, which is
// worth 5 % on the 2^24 workload.
// (Three blocks of the one-dither sink at 40 registers were measured slower, 0.96 against 0.80 ms.)
template <int T, int SINK>
__host__ __device__ constexpr int min_blocks()
{
    return 1 << (15 - T);
}

// The streamed form of that sink spills twice as much at 64 (112 bytes), in its loop: three blocks to an SM in place of four,
// at 80 registers (two workers of 2^23 in 16 blocks 332 -> 322 us, four of 2^20 in 32 150 -> 140, three of 2^27 349 -> 304).
template <int T, int SINK>
__host__ __device__ constexpr int stream_blocks()
{
    if constexpr (SINK == SINK_FINAL && T <= 13) return 3 << (13 - T);
    else return min_blocks<T, SINK>();
}

// ---- the three rounds on the padded tile ---------------------------------------------------
// registers g * 2^VB .. + 2^VB - 1 of round F are consecutive coordinates starting at this tile offset
template <int T>
__device__ __forceinline__ constexpr int round_F_offset(int g) { return reg_offset(RowCfg<T>::FMASK, g << RowCfg<T>::VB); }

template <int T>
__device__ __forceinline__ void store_round_F(float* smem, int baseF, const float (&v)[32])
{
    constexpr int VB = RowCfg<T>::VB;
    float* const pf = smem + phys(baseF);   // (the lane's low coordinate bits never carry into the register bits)
#pragma unroll
    for (int g = 0; g < (32 >> VB); ++g) {
        float* const q = pf + phys(round_F_offset<T>(g));
        if constexpr (VB == 2) *reinterpret_cast<float4*>(q) = make_float4(v[4 * g + 0], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]);
        else if constexpr (VB == 1) *reinterpret_cast<float2*>(q) = make_float2(v[2 * g + 0], v[2 * g + 1]);
        else *q = v[g];
    }
}

// this warp's 1024 coordinates: lane = bits 5..9, registers = bits 0..4
template <int T>
__device__ __forceinline__ void round_M(float* smem, int baseM, float (&v)[32])
{
    using C = RowCfg<T>;
    float4* const pm = reinterpret_cast<float4*>(smem + phys(baseM));
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const float4 x = pm[q];
        v[4 * q + 0] = x.x; v[4 * q + 1] = x.y; v[4 * q + 2] = x.z; v[4 * q + 3] = x.w;
    }
    butterflies32<C::ACT_M>(v);
#pragma unroll
    for (int q = 0; q < 8; ++q) pm[q] = make_float4(v[4 * q + 0], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    __syncwarp();
}

__device__ __forceinline__ void load_round_L(const float* smem, int baseL, float (&v)[32])
{
    const float* const pl = smem + phys(baseL);
#pragma unroll
    for (int r = 0; r < 32; ++r) v[r] = pl[phys(r << 5)];
}

// ---- sinks: register r holds coordinate i0 + 32 r, lane = coordinate & 31 --------------------
__device__ __forceinline__ void sink_ws(const PassParams& p, int n, int64_t i0, const float (&v)[32])
{
    float* dst = static_cast<float*>(p.dst) + (int64_t)n * p.dst_stride + i0;
#pragma unroll
    for (int r = 0; r < 32; ++r) dst[r << 5] = v[r] * p.scale;
}

// Sign bits are shifted into a per-lane mask (bit r = sign of register r), then the 32 x 32 bit
// matrix is transposed across the warp so that lane r owns packed word r.
// EARLY: the words were left at early[0], early[stride], ..
template <bool EARLY = false>
__device__ __forceinline__ void sink_pack1(const PassParamsRK& p, int n, uint32_t id, int64_t i0, uint32_t lane,
                                           const float (&v)[32], float amp, const uint4* early = nullptr, int stride = 0)
{
    const uint32_t cbase = ((uint32_t)(i0 >> 7) << 5) + lane;
    const float dc = p.dither_c * amp;
    const float c2 = 2.f * dc, c0 = -16777215.f * dc;
    uint32_t neg = 0;
#pragma unroll
    for (int m = 7; m >= 0; --m) {
        const uint4 w = EARLY ? early[m * stride] : rng_words_dither(p, id, 1u, cbase + 32u * m);
        const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int q = 3; q >= 0; --q) {
            // z = (2 k24 + 1 - 2^24) c + y, k24 = top 24 bits of the word (two roundings: the two operations
            // are independent of each other's latency, 4 % faster than the single-rounding form of the
            // K-dither sink, and with one dither per coordinate the ties stay far inside the allowance)
            const float z = fmaf((float)(ww[q] >> 8), c2, v[4 * m + q] + c0);
            neg = __funnelshift_l(__float_as_uint(z), neg, 1);  // neg = neg << 1 | sign(z)
        }
    }
    const uint32_t mine = warp_transpose_bits(~neg, lane);
    uint32_t* dst = static_cast<uint32_t*>(p.dst) + (int64_t)n * p.dst_stride;
    dst[((i0 - lane) >> 5) + lane] = mine;
}

// K dithers: the count c_r of non-negative signs of register r is kept bit-sliced, plane b being a
// per-lane word whose bit r is bit b of c_r.  Each dither yields the sign mask of the 32 registers
// (funnel shifts, as above), which a ripple of AND/XOR adds to the planes; at the end every plane
// goes through the same warp transpose as the one-dither sink.  No per-register counters.
__device__ __forceinline__ void sink_packK(const PassParamsRK& p, int n, uint32_t id, int64_t i0, uint32_t lane,
                                           const float (&v)[32], float amp)
{
    const uint32_t cbase = ((uint32_t)(i0 >> 7) << 5) + lane;
    const float dc = p.dither_c * amp;
    uint32_t plane[8];
#pragma unroll
    for (int b = 0; b < 8; ++b) plane[b] = 0u;
    for (int k = 0; k < p.K; ++k) {
        uint32_t neg = 0;
#pragma unroll
        for (int m = 7; m >= 0; --m) {
            const uint4 w = rng_words_dither(p, id, 1u + (uint32_t)k, cbase + 32u * m);
            const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int q = 3; q >= 0; --q) {
                const float z = fmaf(fmaf((float)(ww[q] >> 8), 2.f, -16777215.f), dc, v[4 * m + q]);
                neg = __funnelshift_l(__float_as_uint(z), neg, 1);
            }
        }
        uint32_t carry = ~neg;   // bit r: register r counts one more
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            if (b < p.P) {
                const uint32_t t = plane[b] & carry;
                plane[b] ^= carry;
                carry = t;
            }
        }
    }
    uint32_t* dst = static_cast<uint32_t*>(p.dst) + (int64_t)n * p.dst_stride + ((i0 - lane) >> 5) + lane;
#pragma unroll
    for (int b = 0; b < 8; ++b)
        if (b < p.P) dst[(int64_t)b * (p.dp >> 5)] = warp_transpose_bits(plane[b], lane);
}

__device__ __forceinline__ void sink_final_store(const PassParams& p, int64_t i0, const float (&accv)[32], float amp)
{
    float* const dst = static_cast<float*>(p.dst) + i0;
    const float sc = p.scale * amp;
    const int64_t left = p.d_out - i0;
    if (p.overwrite == 1) {
#pragma unroll
        for (int r = 0; r < 32; ++r)
            if ((r << 5) < left) dst[r << 5] = accv[r] * sc;
    } else {
        // read-modify-write, eight loads in flight at a time
#pragma unroll
        for (int q = 0; q < 32; q += 8) {
            float c[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) c[r] = ((q + r) << 5) < left ? dst[(q + r) << 5] : 0.f;
#pragma unroll
            for (int r = 0; r < 8; ++r)
                if (((q + r) << 5) < left) dst[(q + r) << 5] = p.overwrite == 2 ? fmaf(accv[q + r], sc, c[r]) : (accv[q + r] + c[r]) * sc;
        }
    }
}

// the same for a tile whose workers were shared among the blocks of a cluster
template <int T>
__device__ __forceinline__ void split_final_store(const PassParams& p, int64_t tile_base, int baseL, float* smem,
                                                  const float (&accv)[32], float amp)
{
    __syncthreads();   // the exchange tile is free
#pragma unroll
    for (int r = 0; r < 32; ++r) smem[baseL + (r << 5)] = accv[r];
    cluster_reduce_store<T>(p, tile_base, smem, blockIdx.y, gridDim.y, p.scale * amp, [](uint32_t e) { return e; });
}

// ---- round F's registers from memory ----------------------------------------------------------
// A tile of the gradient, zeros beyond its end.  WHOLE: the end lies elsewhere.  bf16 is widened after the last load:
// behind the bounds checks each widening would otherwise make the next load wait.
template <int T, int SRC, bool WHOLE>
__device__ __forceinline__ void load_gradient_tile(const PassParams& p, int n, int64_t i0, float (&v)[32])
{
    constexpr int VB = RowCfg<T>::VB, VN = 1 << VB, NG = 32 >> VB;
    const int64_t left = p.d - i0;    // valid elements from this thread's first coordinate on
    if constexpr (SRC == SRC_G32) {
        const float* const src = static_cast<const float*>(p.src) + (int64_t)n * p.src_stride + i0;
#pragma unroll
        for (int g = 0; g < NG; ++g) {
            const int o = round_F_offset<T>(g);
            float* const x = v + g * VN;
            if (WHOLE || o + VN <= left) {
                if constexpr (VB == 2) {
                    const float4 q = load_cs(reinterpret_cast<const float4*>(src + o));
                    x[0] = q.x; x[1] = q.y; x[2] = q.z; x[3] = q.w;
                } else if constexpr (VB == 1) {
                    const float2 q = load_cs(reinterpret_cast<const float2*>(src + o));
                    x[0] = q.x; x[1] = q.y;
                } else {
                    x[0] = load_cs(src + o);
                }
            } else {
#pragma unroll
                for (int k = 0; k < VN; ++k) x[k] = (o + k < left) ? src[o + k] : 0.f;
            }
        }
    } else {
        const uint16_t* const src = static_cast<const uint16_t*>(p.src) + (int64_t)n * p.src_stride + i0;
        constexpr int NW = VB == 2 ? 2 : 1;     // 32-bit words of a group
        uint32_t q[NG * NW];
#pragma unroll
        for (int g = 0; g < NG; ++g) {
            const int o = round_F_offset<T>(g);
            uint32_t* const x = q + g * NW;
            if (WHOLE || o + VN <= left) {
                if constexpr (VB == 2) {
                    const uint2 two = load_cs(reinterpret_cast<const uint2*>(src + o));
                    x[0] = two.x; x[1] = two.y;
                } else if constexpr (VB == 1) {
                    x[0] = load_cs(reinterpret_cast<const uint32_t*>(src + o));
                } else {
                    x[0] = load_cs(src + o);
                }
            } else {
#pragma unroll
                for (int k = 0; k < NW; ++k) x[k] = 0u;
#pragma unroll
                for (int k = 0; k < VN; ++k)
                    if (o + k < left) x[k >> 1] |= (uint32_t)src[o + k] << (16 * (k & 1));
            }
        }
#pragma unroll
        for (int r = 0; r < 32; ++r) {
            const uint32_t w = VB == 0 ? q[r] : q[r >> 1];
            v[r] = __uint_as_float((VB > 0 && (r & 1)) ? w & 0xFFFF0000u : w << 16);
        }
    }
}

template <int T, int SRC>
__device__ __forceinline__ void load_gradient(const PassParams& p, int n, int64_t tile_base, int baseF, float (&v)[32])
{
    if (tile_base + ((int64_t)1 << T) <= p.d) load_gradient_tile<T, SRC, true>(p, n, tile_base + baseF, v);
    else load_gradient_tile<T, SRC, false>(p, n, tile_base + baseF, v);
}

// The tile is a whole block of the gradient: its norm sets the block's amplitude, in *s_amp after the next barrier and in
// the table.  One order of the sum (fp64) for every caller.
template <int T>
__device__ __forceinline__ void measure_block(const PassParams& p, int n, int tid, const float (&v)[32], float* s_amp)
{
    __shared__ double wsum[RowCfg<T>::NT / 32];
    double sum = sum_of_squares(v);
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
    if ((tid & 31) == 0) wsum[tid >> 5] = sum;
    __syncthreads();
    if (tid == 0) {
        for (int k = 1; k < RowCfg<T>::NT / 32; ++k) sum += wsum[k];
        *s_amp = fmaxf((float)(p.amp_factor * sqrt(sum)), kMinBlockAmplitude);
        p.amp_out[(int64_t)n * p.amp_stride + blockIdx.x] = *s_amp;
    }
}

// the amplitudes alone, for the callers whose encoder does not measure them
template <int T, int SRC>
__global__ void __launch_bounds__(1 << (T - 5), 1 << (15 - T)) row_norm_kernel(const PassParams p)
{
    __shared__ float s_amp;
    pdl_begin();
    float v[32];
    load_gradient<T, SRC>(p, blockIdx.y, (int64_t)blockIdx.x << T, deposit<RowCfg<T>::FMASK, T>(threadIdx.x), v);
    measure_block<T>(p, blockIdx.y, threadIdx.x, v, &s_amp);
}

// SRC_BITS_TOP.  Entry j of tile t after the top stages is sum_s (-1)^popc(s & t) x_s(j) over the 2^5 segments s of the
// transform, x = 2 b - 1: the number of set bits among b_s(j) ^ parity(s & t).  The thread counts 32 entries at once, one
// packed word per segment, by a tree of bit-sliced adders, and leaves the six planes of the counts at top[0], top[NT], ..
template <int K>
__device__ __forceinline__ void add_planes(uint32_t (&a)[6], const uint32_t (&b)[6])   // a += b, planes 0 .. K - 1 each
{
    uint32_t carry = a[0] & b[0];
    a[0] ^= b[0];
#pragma unroll
    for (int k = 1; k < K; ++k) {
        const uint32_t x = a[k], y = b[k];
        a[k] = x ^ y ^ carry;
        carry = (x & y) | (carry & (x | y));
    }
    a[K] = carry;
}
template <int K>
__device__ __forceinline__ void count_words(const uint32_t* w, uint32_t (&sum)[6])      // planes of the count of 2^K words
{
    if constexpr (K == 0) {
        sum[0] = w[0];
    } else {
        uint32_t other[6];
        count_words<K - 1>(w, sum);
        count_words<K - 1>(w + (1 << (K - 1)), other);
        add_planes<K>(sum, other);
    }
}
template <int T>
__device__ __forceinline__ void count_segments(const PassParams& p, int n, int tid, uint32_t* top)
{
    constexpr int NT = RowCfg<T>::NT;
    const uint32_t t = blockIdx.x & 31u;
    // bit s = parity(s & t)
    const uint32_t odd = ((t & 1u) ? 0xAAAAAAAAu : 0u) ^ ((t & 2u) ? 0xCCCCCCCCu : 0u) ^ ((t & 4u) ? 0xF0F0F0F0u : 0u) ^
                         ((t & 8u) ? 0xFF00FF00u : 0u) ^ ((t & 16u) ? 0xFFFF0000u : 0u);
    const uint32_t* const src = static_cast<const uint32_t*>(p.src) + (int64_t)n * p.src_stride + (int64_t)(blockIdx.x >> 5) * (32 * NT) + tid;
    uint32_t w[32], sum[6];
#pragma unroll
    for (int s = 0; s < 32; ++s) w[s] = load_ca(src + s * NT);
#pragma unroll
    for (int s = 0; s < 32; ++s) w[s] ^= (odd >> s) & 1u ? 0xFFFFFFFFu : 0u;
    count_words<kTopStages>(w, sum);
#pragma unroll
    for (int k = 0; k < 6; ++k) top[k * NT + tid] = sum[k];
}

// fw: flip words of the tile (gradient sources).  ONE_PLANE: a packed source known to have a single plane.
template <int T, int SRC, bool ONE_PLANE = false>
__device__ __forceinline__ void load_source(const PassParams& p, int n, int64_t tile_base, int baseF, const uint32_t* fw,
                                            float (&v)[32])
{
    constexpr int VB = RowCfg<T>::VB, VN = 1 << VB;
    const int64_t i0 = tile_base + baseF;
    if constexpr (SRC == SRC_WS_PAIR || SRC == SRC_WS16_PAIR) {
        // x_0 + x_1 of the pair's halves for its first tile, x_0 - x_1 for its second
        static_assert(VB == 1, "tiles of 2^14");
        const bool second = (tile_base >> T) & 1;
        const int64_t at = (int64_t)n * p.src_stride + i0 - (second ? (int64_t)1 << T : 0);
#pragma unroll
        for (int g = 0; g < 16; ++g) {
            const int o = round_F_offset<T>(g);
            float2 a, b;
            if constexpr (SRC == SRC_WS_PAIR) {
                const float* const src = static_cast<const float*>(p.src) + at;
                a = load_cg(reinterpret_cast<const float2*>(src + o));
                b = load_cg(reinterpret_cast<const float2*>(src + o + (1 << T)));
            } else {
                const __half* const src = static_cast<const __half*>(p.src) + at;
                const uint32_t qa = load_cg(reinterpret_cast<const uint32_t*>(src + o)), qb = load_cg(reinterpret_cast<const uint32_t*>(src + o + (1 << T)));
                a = __half22float2(*reinterpret_cast<const __half2*>(&qa));
                b = __half22float2(*reinterpret_cast<const __half2*>(&qb));
            }
            v[2 * g] = second ? a.x - b.x : a.x + b.x;
            v[2 * g + 1] = second ? a.y - b.y : a.y + b.y;
        }
    } else if constexpr (SRC == SRC_G32 || SRC == SRC_G16) {
        load_gradient<T, SRC>(p, n, tile_base, baseF, v);
    } else if constexpr (SRC == SRC_WS) {
        const float* const src = static_cast<const float*>(p.src) + (int64_t)n * p.src_stride + i0;
#pragma unroll
        for (int g = 0; g < (32 >> VB); ++g) {
            const int o = round_F_offset<T>(g);
            float* const x = v + g * VN;
            static_assert(SRC != SRC_WS || VB >= 1, "an intermediate's tiles of 2^15 are pairs of 2^14");
            if constexpr (VB == 2) {
                const float4 q = load_cs(reinterpret_cast<const float4*>(src + o));
                x[0] = q.x; x[1] = q.y; x[2] = q.z; x[3] = q.w;
            } else {
                const float2 q = load_cs(reinterpret_cast<const float2*>(src + o));
                x[0] = q.x; x[1] = q.y;
            }
        }
    } else if constexpr (SRC == SRC_WS16) {
        const __half* const src = static_cast<const __half*>(p.src) + (int64_t)n * p.src_stride + i0;
#pragma unroll
        for (int g = 0; g < (32 >> VB); ++g) {
            const int o = round_F_offset<T>(g);
            float* const x = v + g * VN;
            if constexpr (VB == 2) {
                const uint2 q = load_cs(reinterpret_cast<const uint2*>(src + o));
                const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&q.x));
                const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&q.y));
                x[0] = a.x; x[1] = a.y; x[2] = b.x; x[3] = b.y;
            } else {
                const uint32_t q = load_cs(reinterpret_cast<const uint32_t*>(src + o));
                const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&q));
                x[0] = a.x; x[1] = a.y;
            }
        }
    } else if constexpr (SRC == SRC_BITS_TOP) {
        const uint32_t* const top = fw + (RowCfg<T>::TOP_AT - RowCfg<T>::TILE_WORDS * 4) / 4 + (baseF >> 5);
        const uint32_t pos = (uint32_t)baseF & 31u;
#pragma unroll
        for (int g = 0; g < (32 >> VB); ++g) {
            const uint32_t* const at = top + (round_F_offset<T>(g) >> 5);
#pragma unroll
            for (int k = 0; k < VN; ++k) v[g * VN + k] = -32.f;
            float weight = 2.f;
#pragma unroll
            for (int pl = 0; pl < 6; ++pl, weight += weight) {
                const uint32_t w = at[pl * RowCfg<T>::NT] >> pos;
#pragma unroll
                for (int k = 0; k < VN; ++k)
                    if ((w >> k) & 1u) v[g * VN + k] += weight;
            }
        }
    } else {  // SRC_BITS
        // plane by plane (one of them: +-1), a word per group of consecutive coordinates; no unrolling over the planes: a
        // short vector runs through this code once, and fetching the instructions would cost more than they do
        const uint32_t* src = static_cast<const uint32_t*>(p.src) + (int64_t)n * p.src_stride + ((tile_base + baseF) >> 5);
        const uint32_t pos = (uint32_t)baseF & 31u;      // (the groups are whole words apart)
        constexpr int NG = 32 >> VB;
        uint32_t w[NG];
        if constexpr (ONE_PLANE) {
#pragma unroll
            for (int g = 0; g < NG; ++g) w[g] = load_ca(src + (round_F_offset<T>(g) >> 5)) >> pos;
#pragma unroll
            for (int r = 0; r < 32; ++r) v[r] = ((w[r >> VB] >> (r & (VN - 1))) & 1u) ? 1.f : -1.f;
        } else {
#pragma unroll
            for (int r = 0; r < 32; ++r) v[r] = (float)(-p.K);
            float weight = 2.f;
#pragma unroll 1
            for (int pl = 0; pl < p.P; ++pl, weight += weight, src += p.dp >> 5) {
#pragma unroll
                for (int g = 0; g < NG; ++g) w[g] = load_ca(src + (round_F_offset<T>(g) >> 5)) >> pos;
#pragma unroll
                for (int r = 0; r < 32; ++r)
                    if ((w[r >> VB] >> (r & (VN - 1))) & 1u) v[r] += weight;
            }
        }
    }
    if constexpr (SRC == SRC_G32 || SRC == SRC_G16) {
#pragma unroll
        for (int g = 0; g < (32 >> VB); ++g) {
            const int e0 = baseF | round_F_offset<T>(g);
            const uint32_t w = fw[e0 >> 5];
            const uint32_t pos = (uint32_t)e0 & 31u;
#pragma unroll
            for (int k = 0; k < VN; ++k) v[g * VN + k] = flip_by_bit(v[g * VN + k], w, pos + k);
        }
    }
}

// =============================================================================================
// row_kernel: sources read by the threads themselves (single-pass transforms)
// =============================================================================================
// EARLY: what comes from the generator alone, the first worker's flips and the dither words of SINK_PACK1, is made before the
// wait for the kernel in front (the words kept in shared memory), where a chain of short kernels hides it: server and
// downlink of 2^17, four workers, 16.6 -> 13.8 us, an encode of eight times 2^13 3.6 -> 2.7, of four times 2^16 6.7 -> 4.9.
template <int T, int SRC, int SINK, bool EARLY>
__global__ void __launch_bounds__(1 << (T - 5), min_blocks<T, SINK>()) row_kernel(const typename KernelParams<SINK>::type p)
{
    using C = RowCfg<T>;
    extern __shared__ __align__(16) float smem[];
    pdl_trigger();
    uint32_t* const fw = reinterpret_cast<uint32_t*>(smem + C::TILE_WORDS);

    const int tid = threadIdx.x;
    const uint32_t lane = tid & 31;
    const int64_t tile_base = (int64_t)blockIdx.x << T;
    // SINK_FINAL: the blocks of a cluster (gridDim.y of them, one if the tiles alone fill the chip) take the
    // workers in turn and add up their sums at the end
    constexpr bool kLoopWorkers = (SINK == SINK_FINAL);
    constexpr bool kMeasures = (SRC == SRC_G32 || SRC == SRC_G16) && SINK == SINK_PACK1;
    constexpr bool kFlips = (SRC == SRC_G32 || SRC == SRC_G16 || SINK == SINK_FINAL || SINK == SINK_SINGLE);
    const int n_begin = (int)blockIdx.y;
    const int n_end = kLoopWorkers ? p.nworkers : n_begin + 1;
    const int n_step = kLoopWorkers ? (int)gridDim.y : 1;
    auto flip_words = [&](uint32_t id) {
        if (tid < C::FLIP_WORDS / 4) {
            const uint4 w = rng_words(p.rng, id, 0u, (uint32_t)(tile_base >> 7) + (uint32_t)tid);
            reinterpret_cast<uint4*>(fw)[tid] = w;
        }
    };
    if (EARLY && kFlips) flip_words(p.id0 + (uint32_t)n_begin);
    uint4* const early = reinterpret_cast<uint4*>(reinterpret_cast<char*>(smem) + C::EARLY_AT) + tid;
    if constexpr (EARLY && SINK == SINK_PACK1) {
        const uint32_t cbase = ((uint32_t)((tile_base + deposit<C::LMASK, T>(tid)) >> 7) << 5) + lane;
#pragma unroll 2
        for (int m = 0; m < 8; ++m) early[m * C::NT] = rng_words_dither(p, p.id0 + (uint32_t)n_begin, 1u, cbase + 32u * m);
    }
    pdl_wait();
    // one amplitude per tile (a block of the blocked mode is at least a tile): thread 0 reads it
    // first, so that its latency hides behind the tile load, and parks it in shared memory until
    // the sink (the barriers of the exchange rounds order the two)
    __shared__ float s_amp;
    if (tid == 0) {
        if (SINK == SINK_SINGLE) s_amp = p.amp_mode != AMP_DITHER ? amplitude_at(p, 0, tile_base) : 1.f;
        else s_amp = (!kLoopWorkers || p.amp_mode == AMP_SCALE) ? amplitude_at(p, kLoopWorkers ? 0 : n_begin, tile_base) : 1.f;
    }

    const int baseF = deposit<C::FMASK, T>(tid);
    const int baseM = deposit<C::MMASK, T>(tid);
    const int baseL = deposit<C::LMASK, T>(tid);
    const int64_t i0 = tile_base + baseL;  // coordinate held in register 0 of round L

    float accv[32];
    if (kLoopWorkers) {
#pragma unroll
        for (int r = 0; r < 32; ++r) accv[r] = 0.f;
    }

    for (int n = n_begin; n < n_end; n += n_step) {
        const uint32_t id = p.id0 + (uint32_t)n;
        const float wamp = (kLoopWorkers && p.amp_mode == AMP_WEIGHT) ? amplitude_at(p, n, tile_base) : 1.f;
        if (kFlips) {
            if (kLoopWorkers && !(EARLY && n == n_begin)) __syncthreads();  // previous worker's readers of fw and of the tile
            if (!EARLY || n != n_begin) flip_words(id);
            if constexpr (SRC == SRC_BITS_TOP) count_segments<T>(p, n, tid, reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(smem) + C::TOP_AT));
            __syncthreads();
        }

        float v[32];
        load_source<T, SRC, kLoopWorkers>(p, n, tile_base, baseF, fw, v);   // (uplink planes come one to a worker)
        if constexpr (kMeasures) {
            if (p.amp_out != nullptr) measure_block<T>(p, n, tid, v, &s_amp);   // (its readers are behind the exchange's barrier)
        }
        butterflies32<31>(v);
        store_round_F<T>(smem, baseF, v);
        __syncthreads();
        round_M<T>(smem, baseM, v);
        load_round_L(smem, baseL, v);
        butterflies32<C::ACT_L>(v);

        if constexpr (SINK == SINK_WS) {
            sink_ws(p, n, i0, v);
        } else if constexpr (SINK == SINK_PACK1) {
            sink_pack1<EARLY>(p, n, id, i0, lane, v, s_amp, early, C::NT);
        } else if constexpr (SINK == SINK_PACKK) {
            sink_packK(p, n, id, i0, lane, v, s_amp);
        } else if constexpr (SINK == SINK_SINGLE) {
            const uint32_t* const fwl = fw + ((baseL - (int)lane) >> 5);
            // (as the first of several workers: a weight rounds the term before the scale, and added to zero a flipped zero is +0)
            const float w = p.amp_mode == AMP_WEIGHT ? s_amp : 1.f;
#pragma unroll
            for (int r = 0; r < 32; ++r) v[r] = fmaf(flip_by_bit(v[r], fwl[r], lane), w, 0.f);
            sink_final_store(p, i0, v, p.amp_mode == AMP_WEIGHT ? 1.f : s_amp);
        } else {
            const uint32_t* const fwl = fw + ((baseL - (int)lane) >> 5);
#pragma unroll
            for (int r = 0; r < 32; ++r) accv[r] = fmaf(flip_by_bit(v[r], fwl[r], lane), wamp, accv[r]);
        }
    }
    if constexpr (SINK == SINK_FINAL) {
        if (gridDim.y == 1) sink_final_store(p, i0, accv, s_amp);
        else split_final_store<T>(p, tile_base, baseL, smem, accv, s_amp);
    }
}

// =============================================================================================
// row_packk_kernel: K > 1 dithers on few tiles, or many dithers
// =============================================================================================
// The generator dominates (K calls per four coordinates against three register rounds), so the block transforms its
// tile into shared memory and its warps then share out the tile's (group of 128 coordinates, range of dithers)
// units.  Where the tiles leave the chip idle, gridDim.y blocks transform the same tile and each dithers a part
// of its groups: one vector of 2^13 with K = 255, a single tile, takes 8 us (without the launch 13.5) against 310
// in one block of eight warps with all dithers of 32 coordinates to a lane; 2^20 with K = 255 0.21 ms against 0.51.
// On a full grid row_kernel's in-register sink is the faster one up to about 24 dithers (2^24, K = 3 / 15 / 31:
// 62 / 228 / 445 us against 84 / 244 / 416): it has eight generator calls in flight per lane and no ballots.
constexpr int kManyDithers = 24;

template <int T>
struct PackKCfg {
    static constexpr int THREADS = RowCfg<T>::NT < 256 ? 256 : RowCfg<T>::NT;
    static constexpr int WARPS = THREADS / 32;
    static constexpr int GROUPS = 1 << (T - 7);
    static constexpr int MIN_BLOCKS = 1024 / THREADS;
    static constexpr size_t SMEM_BYTES = RowCfg<T>::SMEM_BYTES + (size_t)WARPS * 128;   // + packed counts of up to WARPS groups
};

template <int T, int SRC>
__global__ void __launch_bounds__(PackKCfg<T>::THREADS, PackKCfg<T>::MIN_BLOCKS) row_packk_kernel(const PassParamsRK p)
{
    using C = RowCfg<T>;
    using K = PackKCfg<T>;
    extern __shared__ __align__(16) float smem[];
    pdl_begin();
    uint32_t* const fw = reinterpret_cast<uint32_t*>(smem + C::TILE_WORDS);
    uint32_t* const counts = fw + C::FLIP_WORDS + 4;
    const int tid = threadIdx.x;
    const uint32_t lane = tid & 31;
    const int warp = tid >> 5;
    const int64_t tile_base = (int64_t)blockIdx.x << T;
    const int n = blockIdx.z;
    const uint32_t id = p.id0 + (uint32_t)n;
    const bool active = K::THREADS == C::NT || tid < C::NT;      // (whole warps)
    const float dc = p.dither_c * amplitude_at(p, n, tile_base);

    if (SRC == SRC_G32) {
        if (tid < C::FLIP_WORDS / 4)
            reinterpret_cast<uint4*>(fw)[tid] = rng_words(p.rng, id, 0u, (uint32_t)(tile_base >> 7) + (uint32_t)tid);
        __syncthreads();
    }
    if (active) {
        const int baseF = deposit<C::FMASK, T>(tid);
        float v[32];
        load_source<T, SRC>(p, n, tile_base, baseF, fw, v);
        butterflies32<31>(v);
        store_round_F<T>(smem, baseF, v);
    }
    __syncthreads();
    if (active) {
        const int baseL = deposit<C::LMASK, T>(tid);
        float v[32];
        round_M<T>(smem, deposit<C::MMASK, T>(tid), v);
        load_round_L(smem, baseL, v);
        butterflies32<C::ACT_L>(v);
        float* const pl = smem + phys(baseL);
#pragma unroll
        for (int r = 0; r < 32; ++r) pl[phys(r << 5)] = v[r];
    }
    counts[tid] = 0u;
    __syncthreads();

    // this block's groups, and how many warps share the dithers of one (all powers of two)
    const int ngroups = K::GROUPS / (int)gridDim.y, g_first = (int)blockIdx.y * ngroups;
    const int share = ngroups < K::WARPS ? K::WARPS / ngroups : 1;
    const int k0 = p.K * (warp % share) / share, k1 = p.K * (warp % share + 1) / share;
    uint32_t* const dst = static_cast<uint32_t*>(p.dst) + (int64_t)n * p.dst_stride + (tile_base >> 5);
    for (int j = warp / share; j < ngroups; j += K::WARPS / share) {
        const int g = g_first + j;
        float y[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) y[r] = smem[phys(128 * g + 32 * r) + (int)lane];
        const uint32_t c = dither_counts<true>(p, id, (((uint32_t)(tile_base >> 7) + (uint32_t)g) << 5) + lane, y, dc, k0, k1);
        if (share == 1) store_count_planes(c, lane, p.P, dst + 4 * g, p.dp >> 5);
        else atomicAdd(counts + 32 * j + (int)lane, c);
    }
    if (share > 1) {
        __syncthreads();
        if (warp < ngroups) store_count_planes(counts[32 * warp + (int)lane], lane, p.P, dst + 4 * (g_first + warp), p.dp >> 5);
    }
}

// =============================================================================================
// row_stream_kernel: tiles of an intermediate (fp32 or fp16) fetched by bulk async copies
// =============================================================================================
// bumped when a bounded wait on a bulk copy gave up (one counter per translation unit that includes this file)
static __device__ int g_async_wait_timeouts;

// one elected thread: announce `bytes` on the barrier and start the copy global -> shared
__device__ __forceinline__ void bulk_load(void* smem_dst, const void* gsrc, uint32_t bytes, uint64_t* bar)
{
    // order this block's earlier generic-proxy accesses to the buffer before the async-proxy write
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(smem_dst)), "l"(gsrc), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

// A streamed tile lands in a buffer of its own beside the padded work tile, so the copy of tile
// k+1 starts as soon as round F has read tile k out of it and runs underneath rounds M and L
// and the sink.  That needs the landing buffer to fit: fp16 tiles, or fp32 tiles up to 2^13.
template <int T, int SRC>
struct StreamCfg {
    using C = RowCfg<T>;
    static constexpr uint32_t kElem = (SRC == SRC_WS16) ? 2u : 4u;
    static constexpr uint32_t kTileBytes = kElem << T;
    static constexpr bool kFits = (SRC == SRC_WS16) || (T <= 13);
    static constexpr size_t SMEM_BYTES = C::SMEM_BYTES + kTileBytes;
};

template <int T, int SRC, int SINK>
__global__ void __launch_bounds__(1 << (T - 5), stream_blocks<T, SINK>()) row_stream_kernel(const typename KernelParams<SINK>::type p, const int64_t ntiles)
{
    using C = RowCfg<T>;
    using S = StreamCfg<T, SRC>;
    pdl_trigger();
    static_assert(SRC == SRC_WS || SRC == SRC_WS16, "streamed sources only");
    extern __shared__ __align__(16) float smem[];
    uint32_t* const fw = reinterpret_cast<uint32_t*>(smem + C::TILE_WORDS);
    uint64_t* const bar = reinterpret_cast<uint64_t*>(fw + C::FLIP_WORDS);
    float* const landing = reinterpret_cast<float*>(bar + 2);
    constexpr uint32_t kElem = S::kElem;
    constexpr uint32_t kTileBytes = S::kTileBytes;

    const int tid = threadIdx.x;
    const uint32_t lane = tid & 31;
    constexpr bool kFinal = (SINK == SINK_FINAL);
    auto flip_words = [&](uint32_t id, int64_t tile_base) {
        if (tid < C::FLIP_WORDS / 4)
            reinterpret_cast<uint4*>(fw)[tid] = rng_words(p.rng, id, 0u, (uint32_t)(tile_base >> 7) + (uint32_t)tid);
    };
    if (kFinal) flip_words(p.id0 + blockIdx.y, (int64_t)blockIdx.x << T);
    pdl_wait();        // (the flips come from the generator alone)
    // SINK_FINAL: this block's tile is fixed, one amplitude scales the sum (AMP_SCALE; parked in shared
    // memory until the store, the barriers of the worker loop order the two) or every worker brings its
    // own weight (AMP_WEIGHT)
    __shared__ float s_amp_final;
    if (tid == 0) s_amp_final = (kFinal && p.amp_mode == AMP_SCALE) ? amplitude_at(p, 0, (int64_t)blockIdx.x << T) : 1.f;
    // work items: SINK_FINAL -> this block's tile for every worker in turn (every gridDim.y-th of them
    //             where the blocks of a cluster share a tile's workers);
    //             otherwise  -> (worker, tile) pairs strided over the grid
    const int64_t nitems = kFinal ? (int64_t)((p.nworkers - (int)blockIdx.y + (int)gridDim.y - 1) / (int)gridDim.y)
                                  : (ntiles * p.nworkers - (int64_t)blockIdx.x + gridDim.x - 1) / gridDim.x;

    const int baseF = deposit<C::FMASK, T>(tid);
    const int baseM = deposit<C::MMASK, T>(tid);
    const int baseL = deposit<C::LMASK, T>(tid);

    auto item_worker = [&](int64_t j) -> int { return kFinal ? (int)(blockIdx.y + j * gridDim.y) : (int)((blockIdx.x + j * gridDim.x) / ntiles); };
    auto item_tile = [&](int64_t j) -> int64_t { return kFinal ? (int64_t)blockIdx.x : (int64_t)((blockIdx.x + j * gridDim.x) % ntiles); };
    auto item_src = [&](int64_t j) -> const char* {
        return static_cast<const char*>(p.src) + ((int64_t)item_worker(j) * p.src_stride + (item_tile(j) << T)) * kElem;
    };

    if (tid == 0) {
        mbar_init(bar, 1);
        if (nitems > 0) bulk_load(landing, item_src(0), kTileBytes, bar);
    }
    __syncthreads();

    float accv[32];
    if (kFinal) {
#pragma unroll
        for (int r = 0; r < 32; ++r) accv[r] = 0.f;
    }
    uint32_t parity = 0;

    for (int64_t j = 0; j < nitems; ++j) {
        const int n = item_worker(j);
        const int64_t tile_base = item_tile(j) << T;
        const int64_t i0 = tile_base + baseL;
        const uint32_t id = p.id0 + (uint32_t)n;
        const float amp = (kFinal && p.amp_mode == AMP_WEIGHT) ? amplitude_at(p, n, tile_base) : 1.f;

        // bounded wait; the block then agrees on the outcome, so that it stops as a whole
        if (!__syncthreads_and(mbar_wait(bar, parity) ? 1 : 0)) {
            // the one copy in flight is the one that did not arrive: a second bounded wait, so that the
            // engine is not left writing into shared memory that the next block of this SM may own
            if (tid == 0) {
                atomicAdd(&g_async_wait_timeouts, 1);
                mbar_wait(bar, parity);
                mbar_inval(bar);
            }
            __syncthreads();
            break;   // (the sums stay incomplete; the blocks of a cluster still meet at its end)
        }
        parity ^= 1u;

        float v[32];
        // round F reads the tile as it arrived (linear) and writes the padded exchange layout
        constexpr int VN = 1 << C::VB;
#pragma unroll
        for (int g = 0; g < (32 >> C::VB); ++g) {
            const int e0 = baseF | round_F_offset<T>(g);
            float* const x = v + g * VN;
            if constexpr (SRC == SRC_WS) {
                static_assert(SRC != SRC_WS || C::VB == 2, "fp32 tiles are streamed up to 2^13");
                const float4 q = *reinterpret_cast<const float4*>(landing + e0);
                x[0] = q.x; x[1] = q.y; x[2] = q.z; x[3] = q.w;
            } else {
                const __half* const h = reinterpret_cast<const __half*>(landing) + e0;
                static_assert(C::VB >= 1, "an intermediate's tiles of 2^15 are pairs of 2^14");
#pragma unroll
                for (int k = 0; k < VN; k += 2) {
                    const float2 a = __half22float2(*reinterpret_cast<const __half2*>(h + k));
                    x[k] = a.x; x[k + 1] = a.y;
                }
            }
        }
        butterflies32<31>(v);
        store_round_F<T>(smem, baseF, v);
        fence_generic_before_async();   // (the landing buffer is only read by the threads, never written)
        __syncthreads();   // round F complete: the landing buffer is free, nobody is in the previous item
        if (tid == 0 && j + 1 < nitems) bulk_load(landing, item_src(j + 1), kTileBytes, bar);
        if (kFinal && j > 0) flip_words(id, tile_base);
        round_M<T>(smem, baseM, v);
        load_round_L(smem, baseL, v);
        __syncthreads();   // the tile lives in registers: the work tile may be overwritten by the next round F
        butterflies32<C::ACT_L>(v);

        if constexpr (SINK == SINK_WS) {
            sink_ws(p, n, i0, v);
        } else {
            const uint32_t* const fwl = fw + ((baseL - (int)lane) >> 5);
#pragma unroll
            for (int r = 0; r < 32; ++r) accv[r] = fmaf(flip_by_bit(v[r], fwl[r], lane), amp, accv[r]);
        }
    }
    if constexpr (kFinal) {
        if (gridDim.y == 1) sink_final_store(p, ((int64_t)blockIdx.x << T) + baseL, accv, s_amp_final);
        else split_final_store<T>(p, (int64_t)blockIdx.x << T, baseL, smem, accv, s_amp_final);
    }
}

// ---- launchers ---------------------------------------------------------------------------------
template <int T, int SRC, int SINK>
cudaError_t launch_row_one(const PassParams& p, cudaStream_t s)
{
    using C = RowCfg<T>;
    const int64_t ntiles = p.dp >> T;
    int sms = 0;
    const cudaError_t e = sm_count(&sms);
    if (e != cudaSuccess) return e;
    // On the way to the dither sink the fp32 tiles are read by the threads themselves: without the persistent
    // grid the blocks of an SM drift apart and one's loads and butterflies fill the gaps of another's generator
    // rounds (2^27 coordinates, T = 10 / 12 / 13: 0.175 / 0.187 / 0.189 ms against 0.215 / 0.213 / 0.225 ms streamed).
    // One worker per tile leaves nothing to stream either.
    constexpr bool kStream = (SRC == SRC_WS16 || SRC == SRC_WS) && (SINK == SINK_FINAL || SINK == SINK_WS) && StreamCfg<T, SRC>::kFits;
    // a few tiles with many workers each (2^13, 8 workers: one tile) would leave most SMs idle
    // (one worker per block instead of two where a decode is little but latency: four vectors of 2^16 7.0 -> 5.1 us, of
    // 2^17 7.9 -> 6.1; of 2^18 11.3 -> 13.1)
    const int share = SRC == SRC_BITS_TOP && T <= 12 ? 2 * p.nworkers : p.nworkers;
    const unsigned split = SINK == SINK_FINAL ? worker_split(ntiles, share, (int64_t)sms * (kStream ? stream_blocks<T, SINK>() : min_blocks<T, SINK>())) : 1u;
    if constexpr (SINK == SINK_PACKK) {
        // parts of the tiles' groups until the blocks fill the chip
        unsigned parts = 1;
        while ((int)parts < PackKCfg<T>::GROUPS && ntiles * p.nworkers * (2 * parts) <= (int64_t)sms * PackKCfg<T>::MIN_BLOCKS) parts *= 2;
        // large tiles on more than half the SMs: transforming each twice costs more than it spreads (128 tiles of 2^14, K = 3 / 15:
        // 15.9 / 40.5 us by two blocks each, 12.4 / 35.1 by one; of 2^13 11.0 / 23.5 and 8.4 / 22.8, but K = 23 30.0 and 33.0)
        const bool whole = 2 * ntiles * p.nworkers > sms && (T == 14 || (T == 13 && p.K <= 16));
        // (on several waves of tiles of 2^10 and 2^11, which leave most threads of row_packk_kernel out of the transform, up to 28 dithers:
        // 2^24 in blocks of 2^10, K = 24, 341 us in registers, 363 shared; 2^21 58 and 48)
        const int64_t threads = ntiles * p.nworkers * C::NT;
        const int many = T <= 11 && threads >= 1 << 18 ? 28 : kManyDithers;
        if (p.K < many && (parts == 1 || whole)) {
            const dim3 grid((unsigned)ntiles, (unsigned)p.nworkers);
            // (short tiles with more than a few dithers crowd up to 2^17 threads: 2^22, K = 15, 66 us and 62)
            return crowds(threads) || (T <= 12 && p.K >= kThresholdDithers && threads == 1 << 17)
                       ? launch<row_kernel<T, SRC, SINK, false>, false>(grid, C::NT, C::SMEM_BYTES, s, 1, kernel_params<SINK>(p))
                       : launch<row_kernel<T, SRC, SINK, false>>(grid, C::NT, C::SMEM_BYTES, s, 1, kernel_params<SINK>(p));
        }
        return launch<row_packk_kernel<T, SRC>>(dim3((unsigned)ntiles, parts, (unsigned)p.nworkers), PackKCfg<T>::THREADS,
                                                PackKCfg<T>::SMEM_BYTES, s, 1, with_round_keys(p));
    } else if constexpr (kStream) {
        int64_t blocks = ntiles;
        if (SINK != SINK_FINAL) {
            blocks = (int64_t)sms * min_blocks<T, SINK>();
            if (blocks > ntiles * p.nworkers) blocks = ntiles * p.nworkers;
        }
        const dim3 grid((unsigned)blocks, split);
        // (in a chain of launches that add to one sum from 2^14 threads on: eight workers of 2^19 with scratch for three 45 us
        // overlapped, 35 not; three in one launch 10.2 and 12.5)
        const int64_t threads = blocks * split * C::NT;
        if (SINK == SINK_FINAL && (crowds(threads) || (threads == 1 << 14 && p.overwrite == 0)))
            return launch<row_stream_kernel<T, SRC, SINK>, false>(grid, C::NT, StreamCfg<T, SRC>::SMEM_BYTES, s, split, kernel_params<SINK>(p), ntiles);
        return launch<row_stream_kernel<T, SRC, SINK>>(grid, C::NT, StreamCfg<T, SRC>::SMEM_BYTES, s, split, kernel_params<SINK>(p), ntiles);
    } else {
        const dim3 grid((unsigned)ntiles, SINK == SINK_FINAL ? split : (unsigned)p.nworkers);
        constexpr size_t kBytes = SRC == SRC_BITS_TOP ? C::TOP_SMEM_BYTES : C::SMEM_BYTES;
        if constexpr (SINK != SINK_WS && (T <= 12 || ((SRC == SRC_G32 || SRC == SRC_G16 || SRC == SRC_BITS || SRC == SRC_BITS_TOP) && T <= 14))) {
            // one block per SM at most, which finds room beside those of the kernel in front: the early form (above).  Behind
            // a strided pass only up to 2^12: with the larger tiles' shared memory the chain lost more than it gained (four
            // workers of 300007, server and downlink: 26.6 -> 28.3 us; of 2^17, tiles of 2^12: 16.6 -> 13.8)
            if (ntiles * grid.y <= sms)
                return launch<row_kernel<T, SRC, SINK, true>>(grid, C::NT, SINK == SINK_PACK1 ? C::EARLY_SMEM_BYTES : kBytes, s, split, kernel_params<SINK>(p));
        }
        // (not for clusters, which are placed together, nor for tiles of 2^14 and 2^15, whose set-up the overlap hides)
        if (SINK == SINK_FINAL && T <= 13 && split == 1 && crowds(ntiles * C::NT))
            return launch<row_kernel<T, SRC, SINK, false>, false>(grid, C::NT, kBytes, s, split, kernel_params<SINK>(p));
        return launch<row_kernel<T, SRC, SINK, false>>(grid, C::NT, kBytes, s, split, kernel_params<SINK>(p));
    }
}

template <int T>
cudaError_t launch_row_T(int src, int sink, const PassParams& p, cudaStream_t s)
{
#define FOSGD_ROW_CASE(SRC_, SINK_) \
    if (src == SRC_ && sink == SINK_) return launch_row_one<T, SRC_, SINK_>(p, s);
    if (sink == SINK_NORM) {
        const dim3 grid((unsigned)(p.dp >> T), (unsigned)p.nworkers);
        return src == SRC_G16 ? launch<row_norm_kernel<T, SRC_G16>>(grid, 1 << (T - 5), 0, s, 1, p)
                              : launch<row_norm_kernel<T, SRC_G32>>(grid, 1 << (T - 5), 0, s, 1, p);
    }
    FOSGD_ROW_CASE(SRC_G32, SINK_WS)
    FOSGD_ROW_CASE(SRC_G16, SINK_WS)
    FOSGD_ROW_CASE(SRC_G32, SINK_PACK1)
    FOSGD_ROW_CASE(SRC_G16, SINK_PACK1)
    FOSGD_ROW_CASE(SRC_G32, SINK_PACKK)
    FOSGD_ROW_CASE(SRC_BITS, SINK_FINAL)
    FOSGD_ROW_CASE(SRC_BITS, SINK_SINGLE)
    if constexpr (T >= 16 - kTopStages && T <= 18 - kTopStages) {
        FOSGD_ROW_CASE(SRC_BITS_TOP, SINK_FINAL)
        FOSGD_ROW_CASE(SRC_BITS_TOP, SINK_SINGLE)
    }
    if constexpr (T <= 14) {     // (an intermediate's tiles of 2^15 are pairs of 2^14)
        FOSGD_ROW_CASE(SRC_WS, SINK_WS)
        FOSGD_ROW_CASE(SRC_WS, SINK_PACK1)
        FOSGD_ROW_CASE(SRC_WS, SINK_PACKK)
        FOSGD_ROW_CASE(SRC_WS, SINK_FINAL)
        FOSGD_ROW_CASE(SRC_WS, SINK_SINGLE)
        FOSGD_ROW_CASE(SRC_WS16, SINK_FINAL)
        FOSGD_ROW_CASE(SRC_WS16, SINK_SINGLE)
    }
    if constexpr (T == 14) {
        FOSGD_ROW_CASE(SRC_WS_PAIR, SINK_WS)
        FOSGD_ROW_CASE(SRC_WS_PAIR, SINK_PACK1)
        FOSGD_ROW_CASE(SRC_WS_PAIR, SINK_PACKK)
        FOSGD_ROW_CASE(SRC_WS_PAIR, SINK_FINAL)
        FOSGD_ROW_CASE(SRC_WS_PAIR, SINK_SINGLE)
        FOSGD_ROW_CASE(SRC_WS16_PAIR, SINK_FINAL)
        FOSGD_ROW_CASE(SRC_WS16_PAIR, SINK_SINGLE)
    }
#undef FOSGD_ROW_CASE
    return cudaErrorInvalidValue;
}

}  // namespace fosgd
