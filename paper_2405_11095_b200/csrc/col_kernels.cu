// Strided pass: A butterfly stages on the index bits [lo, lo + A) of the coordinate, lo >= 10,
// i.e. the Kronecker factor (H_A (x) I_S) with S = 2^lo.  The vector is read as a matrix with
// rows S apart; a warp always covers 32 or 64 consecutive columns of a row, and the row segment of a
// packed source or of the flip vector is one or two words.  Sources: gradients
// (pad + flip), packed bits, or the fp32 intermediate; the sink is the fp32 intermediate
// (in place when source and sink coincide: a block reads its whole tile before writing it).
//
//   A <= 4: a thread holds the 2^A rows of one column in registers; no shared memory.
//   A = 5..8: col2_kernel, 2^A rows x 64 columns, two adjacent columns per thread.
//   A = 9, 10: a tile of 2^A rows x 32 or 16 columns: round F transforms the top five row bits
//           straight from global memory, round L the remaining low row bits after one exchange
//           through shared memory; A = 10 from fp32 gradients: col4.cuh.
#include <cuda.h>   // CUtensorMap and the encode entry point type; the driver is reached through the runtime

#include "col4.cuh"
#include "common.cuh"

namespace fosgd {

// Coordinates inside one worker's vector are below 2^31, so all per-element index arithmetic is
// done on 32-bit offsets from the worker's base pointer (one widening multiply-add per access
// instead of 64-bit shifts, adds and compares).
template <int SRC>
__device__ __forceinline__ float col_load(const PassParams& p, const void* worker_src, uint32_t i, uint32_t d32)
{
    if (SRC == SRC_G32) {
        return (i < d32) ? load_cs(static_cast<const float*>(worker_src) + i) : 0.f;
    } else if (SRC == SRC_G16) {
        return (i < d32) ? __uint_as_float((uint32_t)load_cs(static_cast<const uint16_t*>(worker_src) + i) << 16) : 0.f;
    } else if (SRC == SRC_WS) {
        return static_cast<const float*>(worker_src)[i];
    } else {
        static_assert(SRC == SRC_WS16 || SRC != SRC_BITS, "packed sources are read word by word");
        return __half2float(static_cast<const __half*>(worker_src)[i]);
    }
}

template <int SRC>
__device__ __forceinline__ const void* worker_source(const PassParams& p, int n)
{
    const size_t es = (SRC == SRC_G16 || SRC == SRC_WS16) ? 2 : 4;
    return static_cast<const char*>(p.src) + (size_t)n * (size_t)p.src_stride * es;
}

// x with its sign flipped iff bit (31 - sh) of word is set
__device__ __forceinline__ float flip_shifted(float x, uint32_t word, uint32_t sh)
{
    return __uint_as_float(__float_as_uint(x) ^ ((word << sh) & 0x80000000u));
}

// Packed source: the 32 columns of a row segment are one word per plane.  Lane r fetches the
// word of the r-th row this warp handles (one gather per warp and plane instead of 32 broadcast loads:
// 2^25 coordinates of two planes, ten stages: 174 us with every thread loading its own words), and a bit
// transpose across the warp (five shuffles instead of one per row) hands every lane its columns.
__device__ __forceinline__ uint32_t bits_row_word(const PassParams& p, const void* worker_src, uint32_t irow, int plane)
{
    return load_ca(static_cast<const uint32_t*>(worker_src) + (irow >> 5) + (int64_t)plane * (p.dp >> 5));
}

// Two adjacent columns of sixteen rows: on entry lane 16 h + r holds the word of row r that covers the columns of
// half-warp h; on return bit r is row r of column 2 (lane & 15), bit 16 + r of the column beside it.
__device__ __forceinline__ uint32_t column_pair_bits(uint32_t word, uint32_t lane)
{
    const uint32_t t = warp_transpose_bits(word, lane);
    const uint32_t a = __shfl_sync(0xFFFFFFFFu, t, 2u * (lane & 15u)), b = __shfl_sync(0xFFFFFFFFu, t, 2u * (lane & 15u) + 1u);
    return __byte_perm(a, b, (lane & 16u) ? 0x7632 : 0x5410);
}

// v[r] = 2 c - K of 32 rows from the P count planes of one column (exact): column(pl) = this lane's column of plane pl,
// one bit per row.  fetch(pl) starts the plane's loads one plane ahead.
template <typename Fetch, typename Column>
__device__ __forceinline__ void planes_to_values(const PassParams& p, float (&v)[32], Fetch fetch, Column column)
{
#pragma unroll
    for (int r = 0; r < 32; ++r) v[r] = (float)(-p.K);
    auto next = fetch(0);
    float weight = 2.f;
    for (int pl = 0; pl < p.P; ++pl, weight += weight) {
        const auto mine = next;
        if (pl + 1 < p.P) next = fetch(pl + 1);
        const uint32_t x = column(mine);
#pragma unroll
        for (int r = 0; r < 32; ++r)
            if ((x >> r) & 1u) v[r] += weight;
    }
}

// the sum over a block of W warps, lanes first, to partial[worker * gridDim.x + block]
template <uint32_t W>
__device__ __forceinline__ void leave_block_sum(double sum, double* partial)
{
    __shared__ double wsum[W];
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
    if ((threadIdx.x & 31u) == 0) wsum[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (uint32_t k = 1; k < W; ++k) sum += wsum[k];
        partial[(int64_t)blockIdx.y * gridDim.x + blockIdx.x] = sum;
    }
}

// ---- A = 4, from gradients ----------------------------------------------------------------
// NORM: also leave the sum of squares of each block's gradient entries in partial[worker * gridDim.x + block]
template <int A, int SRC, bool NORM>
__global__ void __launch_bounds__(256) col_small_kernel(const PassParams p, double* const partial)
{
    static_assert(SRC == SRC_G32 || SRC == SRC_G16, "a decoder's first pass of so few stages is colh_small_kernel");
    constexpr int R = 1 << A;
    pdl_trigger();
    const int n = blockIdx.y;
    const uint32_t lane = threadIdx.x & 31;
    const int64_t col = (int64_t)blockIdx.x * 256 + threadIdx.x;
    const uint32_t lo = (uint32_t)(col & (((int64_t)1 << p.lo_log) - 1));
    const uint32_t hi = (uint32_t)(col >> p.lo_log);
    const uint32_t i_first = (hi << (p.lo_log + A)) + lo;  // row 0 of this column
    const uint32_t step = 1u << p.lo_log;
    const uint32_t d32 = (uint32_t)p.d;
    const void* const wsrc = worker_source<SRC>(p, n);

    uint32_t myword = 0;  // flip word of row `lane` (from the generator alone)
    if ((int)lane < R) myword = eps_word(p.rng, p.id0 + (uint32_t)n, ((i_first - lane) + lane * step) >> 5);
    pdl_wait();
    float v[32];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = col_load<SRC>(p, wsrc, i_first + r * step, d32);
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = flip_shifted(v[r], __shfl_sync(0xFFFFFFFFu, myword, r), 31u - lane);
    if constexpr (NORM) leave_block_sum<8>(sum_of_squares<R>(v), partial);
#pragma unroll
    for (int r = R; r < 32; ++r) v[r] = 0.f;
    butterflies32<R - 1>(v);
    float* dst = static_cast<float*>(p.dst) + (int64_t)n * p.dst_stride;
#pragma unroll
    for (int r = 0; r < R; ++r) dst[i_first + r * step] = v[r];
}

// ---- A = 5..8 ----------------------------------------------------------------------------
// 2^A rows x 64 columns, two adjacent columns x sixteen rows per thread: a warp moves 256 contiguous bytes
// of a row per access (128 from bf16), round F has the top four row bits in registers, round L the low four.
// Bound by memory: 2^27 coordinates of fp32 gradients take 0.17 ms at A = 8 (6.3 TB/s of the 6.5 a plain copy
// reaches), where tiles of 16 columns (64-byte segments) took 0.21 ms; with rows megabytes apart (the top pass
// of a 2^31 transform) the segment width decides: 5.8 ms with 64 bytes per row visit at A = 8, 2.9 ms with 256.
// NORM: also leave the sum of squares of each block's gradient entries in partial[worker * gridDim.x + block] (fp64, fixed order)
template <int A, int SRC, bool NORM>
__global__ void __launch_bounds__(2 << A, 512 >> A) col2_kernel(const PassParams p, double* const partial)
{
    extern __shared__ __align__(16) float2 tile2[];
    constexpr uint32_t WARPS = 1u << (A - 4);
    pdl_begin();
    const int n = blockIdx.y;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t w = threadIdx.x >> 5;
    const uint32_t step = 1u << p.lo_log;                         // one row
    const uint32_t d32 = (uint32_t)p.d;
    const void* const wsrc = worker_source<SRC>(p, n);
    float* const dst = static_cast<float*>(p.dst) + (int64_t)n * p.dst_stride;
    constexpr bool kGrad = SRC == SRC_G32 || SRC == SRC_G16;
    const uint32_t seg = blockIdx.x;                              // 64-column segment id
    double sumsq = 0.0;
    const uint32_t lo0 = (seg << 6) & (step - 1u);
    const uint32_t hi = (uint32_t)(((uint64_t)seg << 6) >> p.lo_log);
    const uint32_t i_tile = (hi << (p.lo_log + A)) + lo0;     // row 0, column 0 of the tile
    // round F: rows k = r * WARPS + w
    const uint32_t i_f = i_tile + w * step + 2u * lane;
    const uint32_t step_f = step * WARPS;
    // the two words (flips, or packed signs) of row r belong to lanes r and 16 + r
    const uint32_t iw = i_tile + w * step + (lane & 15u) * step_f + 32u * (lane >> 4);
    const uint32_t from = lane & 16u, bit = (2u * lane) & 31u;
    float v[32];
    if constexpr (SRC == SRC_BITS) {
        float u[32];    // the sixteen rows of the lane's first column, then those of its second
        planes_to_values(p, u, [&](int pl) { return bits_row_word(p, wsrc, iw, pl); },
                             [&](uint32_t mine) { return column_pair_bits(mine, lane); });
#pragma unroll
        for (int r = 0; r < 16; ++r) { v[2 * r] = u[r]; v[2 * r + 1] = u[16 + r]; }
    } else if constexpr (kGrad) {
        // a tile whose last coordinate is inside the gradient: all sixteen loads in flight, no checks
        const bool whole = i_tile + ((1u << A) - 1u) * step + 63u < d32;
        if constexpr (SRC == SRC_G32) {
            auto load2 = [&](int r) {
                const float2 q = load_cs(reinterpret_cast<const float2*>(static_cast<const float*>(wsrc) + i_f + r * step_f));
                v[2 * r] = q.x; v[2 * r + 1] = q.y;
            };
            if (whole) {
#pragma unroll
                for (int r = 0; r < 16; ++r) load2(r);
            } else {
#pragma unroll
                for (int r = 0; r < 16; ++r) {
                    v[2 * r] = v[2 * r + 1] = 0.f;
                    if (i_f + r * step_f + 1u < d32) load2(r);
                }
            }
        } else {
            // raw pairs first: widening each one where it is loaded would make the checked loads wait for one another
            // (2^32 padded coordinates, seven stages, 61% of the rows inside the gradient: 5.34 ms so)
            uint32_t q[16];
            auto load2 = [&](int r) { return load_cs(reinterpret_cast<const uint32_t*>(static_cast<const uint16_t*>(wsrc) + i_f + r * step_f)); };
            if (whole) {
#pragma unroll
                for (int r = 0; r < 16; ++r) q[r] = load2(r);
            } else {
#pragma unroll
                for (int r = 0; r < 16; ++r) {
                    q[r] = 0u;
                    if (i_f + r * step_f + 1u < d32) q[r] = load2(r);
                }
            }
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                v[2 * r] = __uint_as_float(q[r] << 16); v[2 * r + 1] = __uint_as_float(q[r] & 0xFFFF0000u);
            }
        }
        if (!whole && (d32 & 1u)) {       // an odd length ends inside a pair
#pragma unroll
            for (int r = 0; r < 16; ++r)
                if (i_f + r * step_f + 1u == d32) v[2 * r] = col_load<SRC>(p, wsrc, d32 - 1u, d32);
        }
        const uint32_t mine = eps_word(p.rng, p.id0 + (uint32_t)n, iw >> 5);
        const uint32_t sh = 31u - bit;
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const uint32_t word = __shfl_sync(0xFFFFFFFFu, mine, r + (int)from);
            v[2 * r] = flip_shifted(v[2 * r], word, sh);
            v[2 * r + 1] = flip_shifted(v[2 * r + 1], word, sh - 1u);
        }
    } else if constexpr (SRC == SRC_WS) {
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const float2 q = *reinterpret_cast<const float2*>(static_cast<const float*>(wsrc) + i_f + r * step_f);
            v[2 * r] = q.x; v[2 * r + 1] = q.y;
        }
    } else {
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const float2 q = __half22float2(*reinterpret_cast<const __half2*>(static_cast<const __half*>(wsrc) + i_f + r * step_f));
            v[2 * r] = q.x; v[2 * r + 1] = q.y;
        }
    }
    if constexpr (NORM) sumsq = sum_of_squares(v);
    butterflies32<30>(v);
#pragma unroll
    for (int r = 0; r < 16; ++r) tile2[((r * WARPS + w) << 5) + lane] = make_float2(v[2 * r], v[2 * r + 1]);
    __syncthreads();
    // round L: rows k = w * 16 + r (the low A - 4 bits are new)
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const float2 q = tile2[((w * 16u + r) << 5) + lane];
        v[2 * r] = q.x; v[2 * r + 1] = q.y;
    }
    butterflies32<((1 << (A - 4)) - 1) << 1>(v);
    const uint32_t i_l = i_tile + (w * 16u) * step + 2u * lane;
#pragma unroll
    for (int r = 0; r < 16; ++r)
        __stcg(reinterpret_cast<float2*>(dst + i_l + r * step), make_float2(v[2 * r], v[2 * r + 1]));   // L2 only: read next by another kernel
    if constexpr (NORM) leave_block_sum<WARPS>(sumsq, partial);
}

// ---- A = 9, 10 ---------------------------------------------------------------------------
// NORM: as in col2_kernel
template <int A, int SRC, bool NORM>
__global__ void __launch_bounds__(1 << A, 1024 >> A) col_tile_kernel(const PassParams p, double* const partial)
{
    extern __shared__ __align__(16) float smem[];  // 2^A rows x 32 columns
    constexpr int WARPS = 1 << (A - 5);
    pdl_begin();
    const int n = blockIdx.y;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t w = threadIdx.x >> 5;
    const int64_t seg = blockIdx.x;                               // 32-column segment id
    const uint32_t lo0 = (uint32_t)((seg << 5) & (((int64_t)1 << p.lo_log) - 1));
    const uint32_t hi = (uint32_t)((seg << 5) >> p.lo_log);
    const uint32_t i_tile = (hi << (p.lo_log + A)) + lo0;        // row 0, column 0 of the tile
    const uint32_t step = 1u << p.lo_log;                         // one row
    const uint32_t d32 = (uint32_t)p.d;
    const void* const wsrc = worker_source<SRC>(p, n);

    float v[32];
    const uint32_t irow = i_tile + (lane * WARPS + w) * step;     // row lane * WARPS + w: its words are this lane's to fetch
    // round F: rows k = r * WARPS + w  (register bits = top five row bits)
    const uint32_t i_f = i_tile + w * step + lane;
    const uint32_t step_f = step * WARPS;
    if constexpr (SRC == SRC_BITS) {
        planes_to_values(p, v, [&](int pl) { return bits_row_word(p, wsrc, irow, pl); },
                             [&](uint32_t mine) { return warp_transpose_bits(mine, lane); });
    } else {
#pragma unroll
        for (int r = 0; r < 32; ++r) v[r] = col_load<SRC>(p, wsrc, i_f + r * step_f, d32);
        if (SRC == SRC_G32 || SRC == SRC_G16) {
            const uint32_t mine = eps_word(p.rng, p.id0 + (uint32_t)n, irow >> 5);
#pragma unroll
            for (int r = 0; r < 32; ++r) v[r] = flip_shifted(v[r], __shfl_sync(0xFFFFFFFFu, mine, r), 31u - lane);
        }
    }
    double sumsq = 0.0;
    if constexpr (NORM) sumsq = sum_of_squares(v);
    butterflies32<31>(v);
#pragma unroll
    for (int r = 0; r < 32; ++r) smem[((r * WARPS + w) << 5) + lane] = v[r];
    __syncthreads();
    // round L: rows k = w * 32 + r  (register bits = low five row bits; those below A-5 are new)
#pragma unroll
    for (int r = 0; r < 32; ++r) v[r] = smem[((w * 32 + r) << 5) + lane];
    butterflies32<(A >= 10) ? 31 : ((1 << (A - 5)) - 1)>(v);
    float* const dst = static_cast<float*>(p.dst) + (int64_t)n * p.dst_stride;
    const uint32_t i_l = i_tile + (w * 32) * step + lane;
#pragma unroll
    for (int r = 0; r < 32; ++r) __stcg(dst + i_l + r * step, v[r]);   // L2 only: read next by another kernel
    if constexpr (NORM) leave_block_sum<WARPS>(sumsq, partial);
}

// ---- A > 5, 16-column tiles ----------------------------------------------------------------
// Same two rounds on a tile of 2^A rows x 16 columns (half the shared memory, so two blocks fit
// on an SM and one block's loads overlap the other's arithmetic and stores).  A lane is a
// (column, row-bit) pair: in round F the row bit is bit 0 of the row, in round L bit 5, so a warp
// instruction always touches two rows x 64 contiguous bytes.  Shared memory holds element
// (row k, column c) at word k*16 + c, plus 16 words of padding per 512 (keeps round L, whose two
// half-warps sit 512 words apart, off the same banks).
__host__ __device__ constexpr int phys16(int e) { return e + ((e >> 9) << 4); }

template <int A, int SRC>
__global__ void __launch_bounds__(1 << (A - 1), 2) col_tile16_kernel(const PassParams p)
{
    extern __shared__ __align__(16) float smem[];
    pdl_begin();
    const int n = blockIdx.y;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t c = lane & 15, h = lane >> 4;
    const uint32_t w = threadIdx.x >> 5;
    const int64_t seg = blockIdx.x;                               // 16-column segment id
    const uint32_t lo0 = (uint32_t)((seg << 4) & (((int64_t)1 << p.lo_log) - 1));
    const uint32_t hi = (uint32_t)((seg << 4) >> p.lo_log);
    const uint32_t i_tile = (hi << (p.lo_log + A)) + lo0;        // row 0, column 0 of the tile
    const uint32_t step = 1u << p.lo_log;                         // one row
    const uint32_t d32 = (uint32_t)p.d;
    const uint32_t bitpos = (lo0 & 31u) + c;                      // this lane's bit inside a packed/flip word
    const void* const wsrc = worker_source<SRC>(p, n);

    float v[32];
    // Per-row words (flip word of a gradient row, or the packed signs of a source row):
    // lane j fetches them for rows (r = j & 15, h = j >> 4) and (r = 16 + (j & 15), h = j >> 4); lanes of a
    // half-warp (same h) read the word from lane r & 15 of their own half.
    const uint32_t row_a = ((lane & 15u) << (A - 5)) | (w << 1) | h;
    const uint32_t ia = i_tile + row_a * step, ib = ia + (step << (A - 1));
    // round F: rows k = (r << (A-5)) | (w << 1) | h
    const uint32_t i_f = i_tile + ((w << 1) | h) * step + c;
    const uint32_t step_f = step << (A - 5);
    if constexpr (SRC == SRC_BITS) {
        planes_to_values(p, v, [&](int pl) { return make_uint2(bits_row_word(p, wsrc, ia, pl), bits_row_word(p, wsrc, ib, pl)); },
                             [&](uint2 mine) {
                                 const uint32_t a = __shfl_sync(0xFFFFFFFFu, warp_transpose_bits(mine.x, lane), bitpos);
                                 const uint32_t b = __shfl_sync(0xFFFFFFFFu, warp_transpose_bits(mine.y, lane), bitpos);
                                 return __byte_perm(a, b, h ? 0x7632 : 0x5410);
                             });
    } else {
        // (flip words first and every flip beside its load: bf16, 4 x 2^24, 122 us; words made behind the loads 135)
        uint32_t word_lo = 0, word_hi = 0;
        if (SRC == SRC_G32 || SRC == SRC_G16) {
            word_lo = eps_word(p.rng, p.id0 + (uint32_t)n, ia >> 5);
            word_hi = eps_word(p.rng, p.id0 + (uint32_t)n, ib >> 5);
        }
        auto load_rows = [&](const uint32_t bound) {
#pragma unroll
            for (int r = 0; r < 32; ++r) {
                v[r] = col_load<SRC>(p, wsrc, i_f + r * step_f, bound);
                if (SRC == SRC_G32 || SRC == SRC_G16)
                    v[r] = flip_shifted(v[r], __shfl_sync(0xFFFFFFFFu, r < 16 ? word_lo : word_hi, r & 15, 16), 31u - bitpos);
            }
        };
        // a block whose last coordinate is inside the gradient needs no per-element bound check
        // (the constant bound folds the checks away)
        if (i_tile + (((1u << A) - 1u) * step) + 15u < d32) load_rows(0xFFFFFFFFu);
        else load_rows(d32);
    }
    butterflies32<31>(v);
    {
        float* const pf = smem + phys16((int)((((w << 1) | h) << 4) + c));
#pragma unroll
        for (int r = 0; r < 32; ++r) pf[phys16(r << (A - 1))] = v[r];
    }
    __syncthreads();
    // round L: rows k = (w << 6) | (h << 5) | r
    {
        const float* const pl = smem + phys16((int)((((w << 6) | (h << 5)) << 4) + c));
#pragma unroll
        for (int r = 0; r < 32; ++r) v[r] = pl[r << 4];
    }
    butterflies32<(A >= 10) ? 31 : ((1 << (A - 5)) - 1)>(v);
    float* const dst = static_cast<float*>(p.dst) + (int64_t)n * p.dst_stride;
    const uint32_t i_l = i_tile + ((w << 6) | (h << 5)) * step + c;
#pragma unroll
    for (int r = 0; r < 32; ++r) __stcg(dst + i_l + r * step, v[r]);   // L2 only: read next by another kernel
}

// ---- A = 10, gradients or the fp32 intermediate: tiles staged by the tensor copy engine (col4.cuh) ----
static __device__ int g_col_wait_timeouts;   // groups that abandoned a bounded wait

__global__ void __launch_bounds__(512, 2) col4_kernel(const PassParams p, const __grid_constant__ CUtensorMap tmap,
                                                      const int nruns, const uint32_t full_rows)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    pdl_begin();
    col4_run<BlockSync>(p, &tmap, full_rows, (int)(blockIdx.x / (unsigned)nruns), (blockIdx.x % (unsigned)nruns) * 8u, smem_raw,
                        (int)threadIdx.x, &g_col_wait_timeouts);
}

// the same, also leaving the sum of squares of every run's gradient entries in partial[worker * nruns + run]
__global__ void __launch_bounds__(512, 2) col4_norm_kernel(const PassParams p, const __grid_constant__ CUtensorMap tmap,
                                                           const int nruns, const uint32_t full_rows, double* const partial)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    pdl_begin();
    col4_run<BlockSync, true>(p, &tmap, full_rows, (int)(blockIdx.x / (unsigned)nruns), (blockIdx.x % (unsigned)nruns) * 8u, smem_raw,
                              (int)threadIdx.x, &g_col_wait_timeouts, partial + blockIdx.x);
}

__global__ void __launch_bounds__(1024, 1) col4_duo_kernel(const PassParams p, const __grid_constant__ CUtensorMap tmap,
                                                           const int nruns, const uint32_t full_rows)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    pdl_begin();
    col4_duo(p, &tmap, (uint32_t)nruns, full_rows, (uint32_t)nruns * (uint32_t)p.nworkers, smem_raw, &g_col_wait_timeouts);
}

cudaError_t col_timeouts(int* out) { return cudaMemcpyFromSymbol(out, g_col_wait_timeouts, sizeof(int)); }

// Tensor map over the gradients as the strided pass sees them: (S columns, whole rows, workers).
// False if the driver entry point is missing or refuses the geometry; the caller then uses the plain kernel.
bool make_col_tensor_map(CUtensorMap* map, const void* base, uint64_t S, uint64_t rows, uint64_t workers,
                         uint64_t worker_stride_elems)
{
    using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static EncodeFn encode = []() -> EncodeFn {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return nullptr;
        return reinterpret_cast<EncodeFn>(fn);
    }();
    if (encode == nullptr || rows == 0) return false;
    const cuuint64_t dims[3] = {S, rows, workers};
    const cuuint64_t strides[2] = {S * 4, worker_stride_elems * 4};
    const cuuint32_t box[3] = {16, 256, 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Ten stages on fp32 gradients through the copy engine.  *launched stays false where it does not apply
// (rows shorter than a run of 128 columns, or the driver refuses the map).
static cudaError_t launch_col4(const PassParams& p, cudaStream_t s, bool* launched)
{
    constexpr int A = 10;
    *launched = false;
    const uint64_t S = (uint64_t)1 << p.lo_log;
    const uint64_t rows = (uint64_t)(p.d >> p.lo_log);   // whole rows
    const int64_t nsegs = (p.dp >> A) / 16;
    const int64_t nruns = nsegs / 8;
    if (S < 128 || nsegs % 8 != 0 || nruns * p.nworkers > 0x7FFFFFFF) return cudaSuccess;
    CUtensorMap map;
    if (!make_col_tensor_map(&map, p.src, S, rows, (uint64_t)p.nworkers, (uint64_t)p.src_stride)) return cudaSuccess;
    *launched = true;
    if (p.lo_log >= 15) {
        // rows 128 KiB apart or more: the two-group persistent form (0.44 against 0.48 ms on 8 workers of 2^25)
        int sms = 0;
        const cudaError_t e = sm_count(&sms);
        if (e != cudaSuccess) return e;
        const int64_t runs = nruns * p.nworkers;
        return launch<col4_duo_kernel>(dim3((unsigned)(runs < sms ? runs : sms)), 1024, Col4Duo::SMEM_BYTES, s, 1, p, map, (int)nruns, (uint32_t)rows);
    }
    // one block per run (0.83 against 0.91 ms on 32 workers of 2^24; blocks that start at different times
    // keep the memory system evenly loaded)
    return launch<col4_kernel>(dim3((unsigned)(nruns * p.nworkers)), 512, Col4::SMEM_BYTES, s, 1, p, map, (int)nruns, (uint32_t)rows);
}

template <int A, int SRC, bool NORM>
static cudaError_t launch_col2(const PassParams& p, double* partial, cudaStream_t s)
{
    return launch<col2_kernel<A, SRC, NORM>>(dim3((unsigned)((p.dp >> A) / 64), (unsigned)p.nworkers), 2 << A, (size_t)(1 << A) * 256, s, 1, p, partial);
}

template <int A, int SRC, bool NORM>
static cudaError_t launch_col_tile(const PassParams& p, double* partial, cudaStream_t s)
{
    return launch<col_tile_kernel<A, SRC, NORM>>(dim3((unsigned)((p.dp >> A) / 32), (unsigned)p.nworkers), 1 << A, (size_t)(1 << A) * 128, s, 1, p, partial);
}

// Strided pass on fp32 gradients with the squared norm of every worker's gradient gathered on the way: sums of
// parts in sums[worker][part], *nparts_out (at most 256, what the caller's scratch holds) of them per worker.  A pass of more
// parts leaves them in `room` (8 bytes per 2^11 coordinates at most: the packed words that the next kernel writes take 2^8), for a second
// kernel to add up.  (Blocks that walk tiles 256 apart instead: one worker of 2^25 in blocks of 2^20 187 us, the norm pass of its own 139.)
// *launched stays false where no kernel carries the sums: four stages, rows 128 KiB apart or more at ten, map refused.
cudaError_t launch_col_norm(int A, const PassParams& p, double* sums, double* room, cudaStream_t s, bool* launched, int* nparts_out)
{
    constexpr int64_t kMaxParts = 256;
    *launched = false;
    const int64_t parts = A == 10 ? ((p.dp >> A) / 16) / 8 : (p.dp >> A) / (A == 9 ? 32 : 64);      // runs, tiles
    double* const partial = parts > kMaxParts ? room : sums;
    cudaError_t e;
    if (A == 10) {
        const uint64_t S = (uint64_t)1 << p.lo_log;
        const uint64_t rows = (uint64_t)(p.d >> p.lo_log);
        if (p.lo_log >= 15 || S < 128 || ((p.dp >> A) / 16) % 8 != 0 || parts * p.nworkers > 0x7FFFFFFF) return cudaSuccess;
        CUtensorMap map;
        if (!make_col_tensor_map(&map, p.src, S, rows, (uint64_t)p.nworkers, (uint64_t)p.src_stride)) return cudaSuccess;
        e = launch<col4_norm_kernel>(dim3((unsigned)(parts * p.nworkers)), 512, Col4::SMEM_BYTES, s, 1, p, map, (int)parts, (uint32_t)rows, partial);
    } else {
        switch (A) {
            case 5: e = launch_col2<5, SRC_G32, true>(p, partial, s); break;
            case 6: e = launch_col2<6, SRC_G32, true>(p, partial, s); break;
            case 7: e = launch_col2<7, SRC_G32, true>(p, partial, s); break;
            case 8: e = launch_col2<8, SRC_G32, true>(p, partial, s); break;
            case 9: e = launch_col_tile<9, SRC_G32, true>(p, partial, s); break;
            default: return cudaSuccess;
        }
    }
    *launched = true;
    *nparts_out = (int)(parts > kMaxParts ? kMaxParts : parts);
    return e == cudaSuccess && parts > kMaxParts ? launch_sum_parts(room, parts, p.nworkers, sums, (int)kMaxParts, s) : e;
}

template <int SRC>
static cudaError_t launch_col_block_norm_src(int A, const PassParams& p, double* partial, cudaStream_t s, bool* launched, int64_t* parts)
{
    *launched = true;
    if (A == 4) {
        *parts = (p.dp >> A) / 256;
        return launch<col_small_kernel<4, SRC, true>>(dim3((unsigned)*parts, (unsigned)p.nworkers), 256, 0, s, 1, p, partial);
    }
    *parts = (p.dp >> A) / 64;
    switch (A) {
        case 5: return launch_col2<5, SRC, true>(p, partial, s);
        case 6: return launch_col2<6, SRC, true>(p, partial, s);
        case 7: return launch_col2<7, SRC, true>(p, partial, s);
        case 8: return launch_col2<8, SRC, true>(p, partial, s);
    }
    *launched = false;
    return cudaSuccess;
}

// Tiles never span two transforms and a transform's tiles are numbered one after the other, so a block's sums are
// adjacent.  (At most one sum per 2^11 coordinates: what the scratch of the separate norm pass holds twice over.)
cudaError_t launch_col_block_norm(int A, int src, const PassParams& p, double* partial, cudaStream_t s, bool* launched, int64_t* parts_per_worker)
{
    return src == SRC_G16 ? launch_col_block_norm_src<SRC_G16>(A, p, partial, s, launched, parts_per_worker)
                          : launch_col_block_norm_src<SRC_G32>(A, p, partial, s, launched, parts_per_worker);
}

// ---- packed source, fp16 arithmetic ------------------------------------------------------------
// A decoder's first pass starts from 2 c - K (one plane: +-1), and after A stages every value is an integer of
// magnitude <= K 2^A, which fp16 holds exactly up to 2048.  So this variant keeps two adjacent columns per
// lane as a half2: 64 columns per warp, butterflies are HADD2 (two coordinates
// per instruction), and the intermediate is written as fp16 (half the bytes, still full
// 128-byte lines per warp).  A row segment of the source is two words per plane: lanes fetch them, one
// gather for every sixteen rows, and a bit transpose hands every lane its columns.
// rows 0..15 (a) and 16..31 (b) of two adjacent columns, one bit each as column_pair_bits leaves them, as +-1
__device__ __forceinline__ void signs_to_half2(uint32_t a, uint32_t b, __half2 (&v)[32])
{
#pragma unroll
    for (int r = 0; r < 32; ++r) {
        // bit r -> sign of the low half, bit 16 + r -> sign of the high half; set bit = +1
        const uint32_t hb = 0xBC00BC00u ^ (((r < 16 ? a : b) << (15 - (r & 15))) & 0x80008000u);
        v[r] = *reinterpret_cast<const __half2*>(&hb);
    }
}

// at(r): coordinate of register r = 0 .. 31, column 0 of the warp's 64
template <typename At>
__device__ __forceinline__ void load_planes_half2(const PassParams& p, const uint32_t* bits, uint32_t lane, __half2 (&v)[32], At at)
{
    // words of registers (lane & 15) and 16 + (lane & 15), column half lane >> 4
    const uint32_t* const wa = bits + (at(lane & 15u) >> 5) + (lane >> 4);
    const uint32_t* const wb = bits + (at(16u + (lane & 15u)) >> 5) + (lane >> 4);
    if (p.P == 1) {
        const uint32_t word_a = load_ca(wa), word_b = load_ca(wb);
        signs_to_half2(column_pair_bits(word_a, lane), column_pair_bits(word_b, lane), v);
    } else {
        const __half2 base = __float2half2_rn((float)(-p.K));
#pragma unroll
        for (int r = 0; r < 32; ++r) v[r] = base;
        uint32_t next_a = load_ca(wa), next_b = load_ca(wb);
        uint32_t weight = 0x4000u;                               // fp16 2.0; the exponent grows plane by plane
        for (int pl = 0; pl < p.P; ++pl, weight += 0x400u) {
            const uint32_t a = column_pair_bits(next_a, lane), b = column_pair_bits(next_b, lane);
            if (pl + 1 < p.P) {
                const int64_t off = (int64_t)(pl + 1) * (p.dp >> 5);
                next_a = load_ca(wa + off);
                next_b = load_ca(wb + off);
            }
#pragma unroll
            for (int r = 0; r < 32; ++r) {
                const uint32_t hb = (((r < 16 ? a : b) >> (r & 15)) & 0x00010001u) * weight;
                v[r] = __hadd2(v[r], *reinterpret_cast<const __half2*>(&hb));
            }
        }
    }
}

// A <= 5: a thread's registers hold the 2^A rows of two columns, for 2^(5-A) adjacent 64-column segments
template <int A>
__global__ void __launch_bounds__(256) colh_small_kernel(const PassParams p)
{
    constexpr uint32_t R = 1u << A;
    constexpr int SEG_LOG = 11 - A;                               // columns of a warp: 2^(5-A) segments of 64
    pdl_begin();
    const int n = blockIdx.y;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t seg = blockIdx.x * 8u + (threadIdx.x >> 5);
    if (seg >= (uint32_t)((p.dp >> A) >> SEG_LOG)) return;        // (whole warps)
    const uint32_t lo0 = (seg << SEG_LOG) & ((1u << p.lo_log) - 1u);
    const uint32_t i_tile = ((uint32_t)(((uint64_t)seg << SEG_LOG) >> p.lo_log) << (p.lo_log + A)) + lo0;
    auto at = [&](uint32_t r) { return i_tile + ((r & (R - 1u)) << p.lo_log) + ((r >> A) << 6); };
    __half2 v[32];
    load_planes_half2(p, static_cast<const uint32_t*>(p.src) + (int64_t)n * p.src_stride, lane, v, at);
    butterflies32<R - 1, __half2>(v);
    __half* const dst = static_cast<__half*>(p.dst) + (int64_t)n * p.dst_stride + 2u * lane;
#pragma unroll
    for (int r = 0; r < 32; ++r)
        __stcg(reinterpret_cast<unsigned int*>(dst + at((uint32_t)r)), *reinterpret_cast<const unsigned int*>(&v[r]));
}

// A = 6..9
template <int A>
__global__ void __launch_bounds__(1 << A, 1024 >> A) colh_tile_kernel(const PassParams p)
{
    extern __shared__ __align__(16) uint32_t smemh[];   // [2^A][32] half2 tile
    constexpr int WARPS = 1 << (A - 5);
    pdl_begin();
    const int n = blockIdx.y;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t w = threadIdx.x >> 5;
    const uint32_t seg = blockIdx.x;                              // 64-column segment id
    const uint32_t lo0 = (seg << 6) & ((1u << p.lo_log) - 1u);
    const uint32_t i_tile = ((uint32_t)(((uint64_t)seg << 6) >> p.lo_log) << (p.lo_log + A)) + lo0;
    const uint32_t step = 1u << p.lo_log;

    __half2 v[32];
    load_planes_half2(p, static_cast<const uint32_t*>(p.src) + (int64_t)n * p.src_stride, lane, v,
                      [&](uint32_t r) { return i_tile + (r * WARPS + w) * step; });
    butterflies32<31, __half2>(v);
    __half2* const tile = reinterpret_cast<__half2*>(smemh);
#pragma unroll
    for (int r = 0; r < 32; ++r) tile[((r * WARPS + w) << 5) + lane] = v[r];
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 32; ++r) v[r] = tile[((w * 32 + r) << 5) + lane];
    butterflies32<(1 << (A - 5)) - 1, __half2>(v);
    __half2* const dst = reinterpret_cast<__half2*>(static_cast<__half*>(p.dst) + (int64_t)n * p.dst_stride + i_tile) + lane;
    const uint32_t i_l = (w * 32u) * (step >> 1);
#pragma unroll
    for (int r = 0; r < 32; ++r)
        __stcg(reinterpret_cast<unsigned int*>(dst + i_l + r * (step >> 1)), *reinterpret_cast<const unsigned int*>(&v[r]));   // L2 only: read next by another kernel
}

// A = 10, one plane: 2^A rows x 32 columns (16 half2 lanes x one row bit per lane, like the
// 16-column fp32 variant): half the shared memory and half the threads per block, so two blocks
// share an SM and one block's stores overlap the other's arithmetic.  A row of the packed source
// is one word; lane j fetches the words of rows (r = j & 15, h = j >> 4) and (16 + (j & 15), h).
template <int A>
__global__ void __launch_bounds__(1 << (A - 1), 2) colh_tile32_kernel(const PassParams p)
{
    extern __shared__ __align__(16) uint32_t smemh[];
    pdl_begin();
    const int n = blockIdx.y;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t c2 = lane & 15, h = lane >> 4;
    const uint32_t w = threadIdx.x >> 5;
    const int64_t seg = blockIdx.x;                               // 32-column segment id
    const uint32_t lo0 = (uint32_t)((seg << 5) & (((int64_t)1 << p.lo_log) - 1));
    const uint32_t hi = (uint32_t)((seg << 5) >> p.lo_log);
    const uint32_t i_tile = (hi << (p.lo_log + A)) + lo0;
    const uint32_t step = 1u << p.lo_log;
    const uint32_t* const bits = static_cast<const uint32_t*>(p.src) + (int64_t)n * p.src_stride;

    uint32_t word_lo, word_hi;
    {
        const uint32_t row_a = ((lane & 15u) << (A - 5)) | (w << 1) | h;
        const uint32_t ia = i_tile + row_a * step;
        word_lo = load_ca(bits + (ia >> 5));
        word_hi = load_ca(bits + ((ia + (step << (A - 1))) >> 5));
    }
    __half2 v[32];
    signs_to_half2(column_pair_bits(word_lo, lane), column_pair_bits(word_hi, lane), v);
    butterflies32<31, __half2>(v);
    __half2* const tile = reinterpret_cast<__half2*>(smemh);
    {
        __half2* const pf = tile + phys16((int)((((w << 1) | h) << 4) + c2));
#pragma unroll
        for (int r = 0; r < 32; ++r) pf[phys16(r << (A - 1))] = v[r];
    }
    __syncthreads();
    {
        const __half2* const pl = tile + phys16((int)((((w << 6) | (h << 5)) << 4) + c2));
#pragma unroll
        for (int r = 0; r < 32; ++r) v[r] = pl[r << 4];
    }
    butterflies32<(A >= 10) ? 31 : ((1 << (A - 5)) - 1), __half2>(v);
    __half2* const dst = reinterpret_cast<__half2*>(static_cast<__half*>(p.dst) + (int64_t)n * p.dst_stride);
    const uint32_t i_l = ((i_tile + ((w << 6) | (h << 5)) * step) >> 1) + c2;
    const uint32_t step2 = step >> 1;
#pragma unroll
    for (int r = 0; r < 32; ++r)
        __stcg(reinterpret_cast<unsigned int*>(dst) + i_l + r * step2, *reinterpret_cast<const unsigned int*>(&v[r]));
}

template <int A>
static cudaError_t launch_colh_one(const PassParams& p, cudaStream_t s)
{
    if constexpr (A <= 5) {
        const uint32_t segs = (uint32_t)(p.dp >> 11);
        return launch<colh_small_kernel<A>>(dim3((segs + 7u) / 8u, (unsigned)p.nworkers), 256, 0, s, 1, p);
    } else if constexpr (A <= 9) {
        return launch<colh_tile_kernel<A>>(dim3((unsigned)((p.dp >> A) / 64), (unsigned)p.nworkers), 1 << A, (size_t)(1 << A) * 128, s, 1, p);
    } else {
        return launch<colh_tile32_kernel<A>>(dim3((unsigned)((p.dp >> A) / 32), (unsigned)p.nworkers), 1 << (A - 1),
                                             (size_t)phys16((1 << A) * 16) * 4, s, 1, p);
    }
}

bool colh_applicable(int A, const PassParams& p)
{
    return p.P == 1 ? A >= 2 && A <= 10 : A >= 2 && A <= 9 && (p.K << A) <= 2048;
}

cudaError_t launch_colh(int A, const PassParams& p, cudaStream_t s)
{
    if (!colh_applicable(A, p)) return cudaErrorInvalidValue;
    switch (A) {
        case 2: return launch_colh_one<2>(p, s);
        case 3: return launch_colh_one<3>(p, s);
        case 4: return launch_colh_one<4>(p, s);
        case 5: return launch_colh_one<5>(p, s);
        case 6: return launch_colh_one<6>(p, s);
        case 7: return launch_colh_one<7>(p, s);
        case 8: return launch_colh_one<8>(p, s);
        case 9: return launch_colh_one<9>(p, s);
        case 10: return launch_colh_one<10>(p, s);
    }
    return cudaErrorInvalidValue;
}

template <int A, int SRC>
static cudaError_t launch_col_one(const PassParams& p, cudaStream_t s)
{
    if constexpr (A <= 4) {
        return launch<col_small_kernel<A, SRC, false>>(dim3((unsigned)((p.dp >> A) / 256), (unsigned)p.nworkers), 256, 0, s, 1, p, nullptr);
    } else if constexpr (A <= 8) {
        return launch_col2<A, SRC, false>(p, nullptr, s);
    } else if constexpr (A == 9) {
        // 32 columns: two blocks of 512 threads per SM, 128-byte row segments (0.20 ms on 2^27 coordinates against
        // 0.24 ms with tiles of 16 columns)
        return launch_col_tile<A, SRC, false>(p, nullptr, s);
    } else {
        // ten stages on fp32 gradients: the copy-engine kernels, unless the driver refuses the tensor map
        if constexpr (SRC == SRC_G32) {
            bool launched = false;
            const cudaError_t e = launch_col4(p, s, &launched);
            if (e != cudaSuccess || launched) return e;
        }
        // 16 columns: at 32 a block fills the SM by itself (0.26 ms against 0.22 ms on 2^27 coordinates)
        return launch<col_tile16_kernel<A, SRC>>(dim3((unsigned)((p.dp >> A) / 16), (unsigned)p.nworkers), 1 << (A - 1),
                                                 (size_t)phys16((1 << A) * 16) * 4, s, 1, p);
    }
}

template <int A>
static cudaError_t launch_col_A(int src, const PassParams& p, cudaStream_t s)
{
    switch (src) {
        case SRC_G32: return launch_col_one<A, SRC_G32>(p, s);
        case SRC_G16: return launch_col_one<A, SRC_G16>(p, s);
        case SRC_BITS:       // what launch_colh does not take: many planes, or two strided passes without scratch for fp16
            if constexpr (A == 6 || A >= 8) return launch_col_one<A, SRC_BITS>(p, s);
            break;
        case SRC_WS:         // the second of two strided passes
            if constexpr (A >= 6 && A <= 9) return launch_col_one<A, SRC_WS>(p, s);
            break;
        case SRC_WS16:
            if constexpr (A >= 6 && A <= 9) return launch_col_one<A, SRC_WS16>(p, s);
            break;
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_col(int A, int src, const PassParams& p, cudaStream_t s)
{
    switch (A) {
        case 4: return launch_col_A<4>(src, p, s);
        case 5: return launch_col_A<5>(src, p, s);
        case 6: return launch_col_A<6>(src, p, s);
        case 7: return launch_col_A<7>(src, p, s);
        case 8: return launch_col_A<8>(src, p, s);
        case 9: return launch_col_A<9>(src, p, s);
        case 10: return launch_col_A<10>(src, p, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace fosgd
