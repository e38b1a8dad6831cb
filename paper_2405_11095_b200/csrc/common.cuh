// Shared device helpers and launch parameter blocks of libfosgd (sm_100a).
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

namespace fosgd {

// ---- sources and sinks of a transform pass -------------------------------------------
enum Src : int {
    SRC_G32 = 0,   // caller gradients, fp32: zero padding beyond d, sign flip D_eps
    SRC_G16 = 1,   // caller gradients, bf16 (exact upcast), same padding and flip
    SRC_BITS = 2,  // packed signs / count planes: q_i = 2 c_i - K
    SRC_WS = 3,    // fp32 intermediate of an earlier pass
    SRC_WS16 = 4,  // fp16 intermediate (exact small integers from a packed source)
    // The contiguous pass of a 2^25 transform, whose 15 stages are one more than a tile of 2^14 has: the top one is
    // done while reading, by both tiles of a pair (each reads both halves, the second time out of L2).
    SRC_WS_PAIR = 5,
    SRC_WS16_PAIR = 6,
    // One plane of a transform of 2^(T + kTopStages): the top stages are counts of packed bits, made while reading
    SRC_BITS_TOP = 7
};
constexpr int kTopStages = 5;
enum Sink : int {
    SINK_WS = 0,     // fp32 intermediate (or the scaled transform output of fosgd_flatten)
    SINK_PACK1 = 1,  // dither + sign + pack, K = 1
    SINK_PACKK = 2,  // K dithers, count, P bit planes
    SINK_FINAL = 3,  // flip, sum over the workers of the launch, optional read-modify-write, scale
    SINK_SINGLE = 4, // SINK_FINAL of a launch with one worker: no sums kept in registers
    SINK_NORM = 6    // no transform: the amplitudes of blocks of one tile each (amp_out)
};

struct Rng {
    uint32_t k0, k1;   // Philox key: lo32(seed), hi32(seed) ^ hi32(step)
    uint32_t step_lo;  // counter word 2
};

struct PassParams {
    const void* src;
    void* dst;
    int64_t src_stride;  // elements (grads, ws) or words (bits) between consecutive workers
    int64_t dst_stride;
    int64_t d;           // valid source elements per worker (gradient sources)
    int64_t dp;          // padded length d'
    int64_t d_out;       // SINK_FINAL: outputs written (d for a decoder, d' for the accumulator)
    float scale;         // SINK_WS and SINK_FINAL: multiplier on the stored value
    float dither_c;      // lambda * sqrt(n) * 2^-24: dither integer -> unnormalised transform units
    int P, K;            // bit planes and dithers
    int overwrite;       // SINK_FINAL: 1 = store scale * sum, 0 = store scale * (dst + sum), 2 = dst += scale * sum
    int nworkers;        // workers handled by this launch
    uint32_t id0;        // generator id of the launch's first worker
    int lo_log;          // strided pass: log2 of the stride between butterfly partners
    // Amplitudes resident on the device (null: folded into dither_c / scale on the host).  Worker n,
    // coordinate i reads amp_dev[n * amp_stride + (i >> amp_shift)]: a single entry (stride 0,
    // shift 31) or one entry per worker and block of the blocked mode.  Pack sinks multiply
    // dither_c by it; SINK_FINAL follows amp_mode.
    const float* amp_dev;
    int64_t amp_stride;
    int amp_shift;
    int amp_mode;        // AMP_DITHER, AMP_SCALE or AMP_WEIGHT
    // Single-pass encoder that measures its own amplitudes (a block of the blocked mode is one tile): worker n's block k
    // gets amp_out[n * amp_stride + k] = max(amp_factor * norm of the block, kMinBlockAmplitude).  Null otherwise.
    float* amp_out;
    double amp_factor;
    Rng rng;
};

enum AmpMode {
    AMP_DITHER = 0,  // SINK_FINAL ignores the amplitudes
    AMP_SCALE = 1,   // SINK_FINAL multiplies its scale by worker 0's entry (one amplitude for all workers)
    AMP_WEIGHT = 2   // SINK_FINAL weights every worker's contribution by that worker's entry
};

// Sum of squares of the first N of a thread's values, in fp64 from the first product on (a square of fp32 is exact there): an fp32 square is
// zero below 4e-23 and infinite above 1.8e19, where gradients still have a norm.  Two chains, to halve the latency.
template <int N = 32>
__device__ __forceinline__ double sum_of_squares(const float (&v)[32])
{
    double s0 = 0.0, s1 = 0.0;
#pragma unroll
    for (int r = 0; r < N; r += 2) {
        s0 = fma((double)v[r], (double)v[r], s0);
        s1 = fma((double)v[r + 1], (double)v[r + 1], s1);
    }
    return s0 + s1;
}

// floor of a measured block amplitude: a block of zeros keeps a positive one, so that its sign bits are still decided by
// the dither (and decode to ~0) instead of by the sign of a zero
constexpr float kMinBlockAmplitude = 1e-30f;

// The parameter block of the kernels with a dither sink: PassParams plus the ten round keys of the
// generator (Weyl sequence of the key), computed once on the host.  As kernel parameters they sit in
// the constant bank and feed the round's logic instruction directly, which saves the two additions
// per round that every call would otherwise repeat (4 % of the one-dither pack pass).  The other
// kernels keep the plain block: with the table in it the flip + accumulate kernels, which never use
// it, ran 8 % slower.
struct PassParamsRK : PassParams {
    uint32_t rk0[10], rk1[10];
};

inline PassParamsRK with_round_keys(const PassParams& p)
{
    PassParamsRK r;
    static_cast<PassParams&>(r) = p;
    for (int i = 0; i < 10; ++i) {
        r.rk0[i] = p.rng.k0 + (uint32_t)i * 0x9E3779B9u;
        r.rk1[i] = p.rng.k1 + (uint32_t)i * 0xBB67AE85u;
    }
    return r;
}

// ---- global loads with a cache hint ----------------------------------------------------------------
// (volatile, unlike the header's __ldg family: never moved ahead of the wait for the kernel before, below)
#define FOSGD_LOAD(NAME, HINT)                                                                                              \
    template <typename V>                                                                                                   \
    __device__ __forceinline__ V NAME(const V* p)                                                                           \
    {                                                                                                                       \
        static_assert(sizeof(V) == 2 || sizeof(V) == 4 || sizeof(V) == 8 || sizeof(V) == 16, "2, 4, 8 or 16 bytes");         \
        V out;                                                                                                              \
        if constexpr (sizeof(V) == 2) {                                                                                     \
            asm volatile("ld.global" HINT ".u16 %0, [%1];" : "=h"(*reinterpret_cast<unsigned short*>(&out)) : "l"(p));      \
        } else if constexpr (sizeof(V) == 4) {                                                                              \
            asm volatile("ld.global" HINT ".b32 %0, [%1];" : "=r"(*reinterpret_cast<uint32_t*>(&out)) : "l"(p));            \
        } else if constexpr (sizeof(V) == 8) {                                                                              \
            uint2& w = *reinterpret_cast<uint2*>(&out);                                                                     \
            asm volatile("ld.global" HINT ".v2.b32 {%0, %1}, [%2];" : "=r"(w.x), "=r"(w.y) : "l"(p));                       \
        } else {                                                                                                            \
            uint4& w = *reinterpret_cast<uint4*>(&out);                                                                     \
            asm volatile("ld.global" HINT ".v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w.x), "=r"(w.y), "=r"(w.z), "=r"(w.w) : "l"(p)); \
        }                                                                                                                   \
        return out;                                                                                                         \
    }
FOSGD_LOAD(load_ca, "")      // all caches
FOSGD_LOAD(load_cg, ".cg")   // L2 only
FOSGD_LOAD(load_cs, ".cs")   // read once
#undef FOSGD_LOAD

// 1 when no table is given
__device__ __forceinline__ float amplitude_at(const PassParams& p, int n, int64_t i)
{
    return p.amp_dev ? load_ca(p.amp_dev + (int64_t)n * p.amp_stride + (i >> p.amp_shift)) : 1.f;
}

// ---- Philox4x32-10 (Salmon et al., SC'11), written from the published round function ----
// Two forms of the same ten rounds.  rng_words_dither takes the round keys from a table in the
// parameter bank: for the dither sinks, whose every thread makes eight calls per tile.  rng_words
// advances the key by addition inside the rounds: for the flip words, which a thread generates once
// or twice per tile.
__device__ __forceinline__ uint4 rng_words_dither(const PassParamsRK& p, uint32_t id, uint32_t domain, uint32_t c)
{
    uint32_t c0 = c, c1 = domain, c2 = p.rng.step_lo, c3 = id;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t p0 = (uint64_t)0xD2511F53u * (uint64_t)c0;
        const uint64_t p1 = (uint64_t)0xCD9E8D57u * (uint64_t)c2;
        const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ p.rk0[r];
        const uint32_t n2 = (uint32_t)(p0 >> 32) ^ c3 ^ p.rk1[r];
        c0 = n0;
        c1 = (uint32_t)p1;
        c2 = n2;
        c3 = (uint32_t)p0;
    }
    return make_uint4(c0, c1, c2, c3);
}

__device__ __forceinline__ uint4 rng_words(const Rng& g, uint32_t id, uint32_t domain, uint32_t c)
{
    uint32_t c0 = c, c1 = domain, c2 = g.step_lo, c3 = id, k0 = g.k0, k1 = g.k1;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t p0 = (uint64_t)0xD2511F53u * (uint64_t)c0;
        const uint64_t p1 = (uint64_t)0xCD9E8D57u * (uint64_t)c2;
        const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ k0;
        const uint32_t n2 = (uint32_t)(p0 >> 32) ^ c3 ^ k1;
        c0 = n0;
        c1 = (uint32_t)p1;
        c2 = n2;
        c3 = (uint32_t)p0;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return make_uint4(c0, c1, c2, c3);
}

__device__ __forceinline__ uint32_t pick(const uint4& w, uint32_t j)
{
    return j == 0 ? w.x : (j == 1 ? w.y : (j == 2 ? w.z : w.w));
}

// Word j of the flip vector eps (32 flips, set bit = -1): output j&3 of counter j>>2, domain 0.
__device__ __forceinline__ uint32_t eps_word(const Rng& g, uint32_t id, uint32_t j)
{
    return pick(rng_words(g, id, 0u, j >> 2), j & 3u);
}

__device__ __forceinline__ float flip_by_bit(float x, uint32_t word, uint32_t bit)
{
    return __uint_as_float(__float_as_uint(x) ^ (((word >> bit) & 1u) << 31));
}

// value of coordinate (word, bit) read from P count planes spaced `plane_words` apart: 2c - K
__device__ __forceinline__ float plane_value(const uint32_t* w0, int64_t plane_words, int P, int K,
                                             uint32_t bit)
{
    int c = 0;
    for (int p = 0; p < P; ++p) c |= (int)((load_ca(w0 + (int64_t)p * plane_words) >> bit) & 1u) << p;
    return (float)(2 * c - K);
}

// 32 x 32 bit-matrix transpose across a warp: on entry lane l holds row l (bit r = entry (l, r));
// on return lane l holds column l (bit r = entry (r, l)).  Five exchange rounds.
__device__ __forceinline__ uint32_t warp_transpose_bits(uint32_t x, uint32_t lane)
{
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1) {
        const uint32_t mask = (s == 16) ? 0x0000FFFFu : (s == 8) ? 0x00FF00FFu : (s == 4) ? 0x0F0F0F0Fu
                            : (s == 2) ? 0x33333333u : 0x55555555u;
        const uint32_t y = __shfl_xor_sync(0xFFFFFFFFu, x, s);
        // lanes with bit s clear keep their low halves and take the partner's low halves shifted up
        x = (lane & s) ? ((x & ~mask) | ((y >> s) & mask)) : ((x & mask) | ((y << s) & ~mask));
    }
    return x;
}

// In-register butterflies over the register-index bits selected by ACTIVE (5-bit mask).
template <int ACTIVE, typename V = float>
__device__ __forceinline__ void butterflies32(V (&v)[32])
{
#pragma unroll
    for (int s = 0; s < 5; ++s) {
        if ((ACTIVE >> s) & 1) {
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                if (!(i & (1 << s))) {
                    const V a = v[i], b = v[i | (1 << s)];
                    v[i] = a + b;
                    v[i | (1 << s)] = a - b;
                }
            }
        }
    }
}

// ---- mbarrier helpers (asynchronous copies signal completion on a shared-memory barrier) ----
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// bounded wait for the barrier phase with the given parity; false if it never completed
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity)
{
    for (int it = 0; it < (1 << 22); ++it) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done) : "r"(smem_u32(bar)), "r"(parity) : "memory");
        if (done) return true;
    }
    return false;
}

__device__ __forceinline__ void mbar_inval(uint64_t* bar)
{
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Every thread that touched a shared-memory buffer through ordinary loads and stores runs this
// before the barrier after which one thread hands the buffer to the asynchronous copy engine.
__device__ __forceinline__ void fence_generic_before_async()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// bar.sync / bar.red are the warp-aligned forms: every lane of a warp must arrive together.  The
// code before them has lane-dependent paths (one lane issues the copies, sixteen patch a row, the
// polling loop of a bounded wait ends per lane), and nothing obliges the compiler to have rejoined
// them in front of an opaque asm statement, so the warp is converged explicitly first.
__device__ __forceinline__ void group_sync(int id, int nthreads)
{
    __syncwarp();
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// barrier + AND over the group: every thread learns whether all of them saw `ok`
__device__ __forceinline__ bool group_all(int id, int nthreads, bool ok)
{
    uint32_t all;
    __syncwarp();
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.and.pred q, %2, %3, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
                 : "=r"(all) : "r"((uint32_t)ok), "r"(id), "r"(nthreads) : "memory");
    return all != 0;
}

// ---- thread-block clusters: the blocks of a cluster read each other's shared memory ----------------
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// four floats at shared-memory address `addr` (a multiple of 16) of the cluster's block `rank`
__device__ __forceinline__ float4 ld_cluster4(uint32_t addr, uint32_t rank)
{
    uint32_t remote;
    float4 q;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(addr), "r"(rank));
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(q.x), "=f"(q.y), "=f"(q.z), "=f"(q.w) : "r"(remote) : "memory");
    return q;
}

// the double at shared-memory address `addr` of the cluster's block `rank`
__device__ __forceinline__ double ld_cluster_double(uint32_t addr, uint32_t rank)
{
    uint32_t remote;
    double q;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(addr), "r"(rank));
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(q) : "r"(remote) : "memory");
    return q;
}

// SINK_FINAL / SINK_SINGLE: one finished sum to memory (sc = scale times amplitude)
__device__ __forceinline__ void store_final(float* dst, float o, float sc, int overwrite)
{
    if (overwrite == 2) {
        *dst = fmaf(o, sc, *dst);   // dst += scale * sum (the descent step on top of the decoder)
    } else {
        if (!overwrite) o += *dst;
        *dst = o * sc;
    }
}

__device__ __forceinline__ void store_final4(float* dst, float4 o, float sc, int overwrite)
{
    float4* const d4 = reinterpret_cast<float4*>(dst);
    if (overwrite == 2) {
        const float4 c = *d4;
        o = make_float4(fmaf(o.x, sc, c.x), fmaf(o.y, sc, c.y), fmaf(o.z, sc, c.z), fmaf(o.w, sc, c.w));
    } else {
        if (!overwrite) {
            const float4 c = *d4;
            o.x += c.x; o.y += c.y; o.z += c.z; o.w += c.w;
        }
        o.x *= sc; o.y *= sc; o.z *= sc; o.w *= sc;
    }
    *d4 = o;
}

// The blocks of a cluster have each left their workers' sums of one tile of 2^T coordinates in shared memory at
// `sums` (`at(e)` = word offset of coordinate e, whole groups of four together); block `rank` of `size` adds its
// share of the coordinates over the blocks in order and stores it.  All threads of all blocks call it.
template <int T, typename At>
__device__ __forceinline__ void cluster_reduce_store(const PassParams& p, int64_t tile_base, const float* sums, uint32_t rank,
                                                     uint32_t size, float sc, At at)
{
    cluster_sync();
    const uint32_t share = (1u << T) / size, base = smem_u32(sums);
    float* const dst = static_cast<float*>(p.dst) + tile_base;
    for (uint32_t e = rank * share + 4u * threadIdx.x; e < (rank + 1u) * share; e += 4u * blockDim.x) {
        float4 o = ld_cluster4(base + 4u * at(e), 0u);
        for (uint32_t k = 1; k < size; ++k) {
            const float4 q = ld_cluster4(base + 4u * at(e), k);
            o.x += q.x; o.y += q.y; o.z += q.z; o.w += q.w;
        }
        const int64_t left = p.d_out - (tile_base + e);
        if (left >= 4) {
            store_final4(dst + e, o, sc, p.overwrite);
        } else {
            if (left > 0) store_final(dst + e, o.x, sc, p.overwrite);
            if (left > 1) store_final(dst + e + 1, o.y, sc, p.overwrite);
            if (left > 2) store_final(dst + e + 2, o.z, sc, p.overwrite);
        }
    }
    cluster_sync();   // nobody leaves while its sums are being read
}

// ---- launching ---------------------------------------------------------------------------------
// Every kernel that goes through launch() may be put on the SMs while its predecessor in the stream is still draining,
// and touches no global memory before pdl_wait(), which returns when the predecessor has completed and its writes
// are visible.  (Its predecessor waited in turn, so everything before it has completed too.)  pdl_trigger() lets the
// successor do the same once every block of this grid has started.  Chains of eight kernels: 2^16 x 4 36.9 -> 31.3 us,
// 2^20 x 16 98.0 -> 90.6.  In a grid launched this way every block pays for its wait, also those that start long
// after the predecessor is gone, so grids of more than kOverlapThreads (1.7 times what the chip holds at once)
// are launched the ordinary way: 25,557,032 x 8 in blocks 985 us with the limit at 10^5 or 3 10^5 threads,
// 993 at 10^6 and 1118 without one; 2^24 x 32 2292, 2288 and 2353; 2^20 x 16, whose kernels have 2^18 and 2^19 threads,
// 95.0, 90.6 and 90.6; one worker of 25,557,032 with a kernel of 2^20 threads 218 without it and 230 with it.  (Kernels
// of short blocks are compiled a second time without the two instructions, for such grids: launch_either.)
constexpr int64_t kOverlapThreads = 1 << 19;
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_begin()
{
    pdl_trigger();
    pdl_wait();
}

// One kernel launch.  Dynamic shared memory beyond the default is allowed once per kernel and device (a driver
// attribute, cheaper to remember than to set before every launch); cluster > 1: clusters of that many blocks in y.
template <auto Kern, bool OVERLAP = true, typename... Args>
inline cudaError_t launch(dim3 grid, unsigned threads, size_t smem, cudaStream_t s, unsigned cluster, const Args&... args)
{
    static std::atomic<uint64_t> allowed{0};   // bit = device
    cudaError_t e;
    if (smem > 48 * 1024) {
        int dev = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
        const uint64_t bit = dev < 64 ? (uint64_t)1 << dev : 0;
        if (!(allowed.load(std::memory_order_acquire) & bit) || bit == 0) {
            if ((e = cudaFuncSetAttribute(Kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
            allowed.fetch_or(bit, std::memory_order_release);
        }
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = OVERLAP && (int64_t)grid.x * grid.y * grid.z * threads <= kOverlapThreads;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 1;
    attr[1].val.clusterDim.y = cluster;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, Kern, args...);
}

// A kernel compiled with and without its wait: overlapped up to `limit` threads, and beyond launched the ordinary way without the
// instruction, which short blocks feel (amplitudes of 2^25 in blocks of 32: 377 us with it, 358 without).
template <auto Overlapped, auto Plain, typename... Args>
inline cudaError_t launch_either(dim3 grid, unsigned threads, cudaStream_t s, int64_t limit, const Args&... args)
{
    return (int64_t)grid.x * grid.y * grid.z * threads <= limit ? launch<Overlapped>(grid, threads, 0, s, 1, args...)
                                                                : launch<Plain, false>(grid, threads, 0, s, 1, args...);
}

inline cudaError_t sm_count(int* sms)
{
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    return e != cudaSuccess ? e : cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
}

// Blocks (a power of two, at most the eight of a portable cluster) that share the workers of one tile, when
// `tiles` blocks alone would leave the chip idle: as many as fit beside each other, at least two workers each.  Starting
// clusters has its price, so that more than 1024 blocks take at least four workers each and there are never more than 2048
// (2^20 cut into tiles of 2^10, four workers: 19 us by pairs, 13 alone; 2^21 in blocks of 2^10, 16: 59 and 53; in blocks of
// 2^11, eight: 25 and 31).
inline unsigned worker_split(int64_t tiles, int nworkers, int64_t resident_blocks)
{
    unsigned s = 1;
    while (s < 8 && tiles * (2 * s) <= resident_blocks && nworkers >= (int)(4 * s) &&
           (tiles * (2 * s) <= 1024 || (tiles * (2 * s) <= 2048 && nworkers >= (int)(8 * s)))) s *= 2;
    return s;
}

// A grid of more than a block per SM and less than a wave, launched while the kernel in front drains, crowds on the SMs that
// have room at that moment and takes longer than it gains, where its blocks take long (row_stream_kernel, two workers of 2^20 16.5 us and
// 10.5 launched the ordinary way; three 21.3 and 12.9; 15 dithers of 2^20 in tiles of 2^11 55 and 30).
inline bool crowds(int64_t threads) { return threads > 1 << 14 && threads < 1 << 17; }

// ---- shared by the translation units of the C-ABI (not exported) -----------------------------
// thread-local last CUDA error behind fosgd_last_cuda_error()
__attribute__((visibility("hidden"))) void set_last_cuda_error(int e);
// argument checks of fosgd_decode without the scratch: FOSGD_OK, FOSGD_EINVAL, FOSGD_EALIGN or FOSGD_EUNSUPPORTED
__attribute__((visibility("hidden"))) int check_decode_args(const void* bits, int64_t d, float lambda, int block_log2,
                                                            const void* out);

// ---- host-visible launchers (one translation unit per family) --------------------------
cudaError_t launch_row(int T, int src, int sink, const PassParams& p, cudaStream_t s);
// one-plane encoder of blocks of 2^16 in one kernel (cluster_encode.cu)
bool cluster_encode_applicable(int L, int64_t dp);
cudaError_t launch_cluster_encode(int src, const PassParams& p, cudaStream_t s);
cudaError_t launch_col(int A, int src, const PassParams& p, cudaStream_t s);
bool colh_applicable(int A, const PassParams& p);                          // every value after A stages exact in fp16
cudaError_t launch_colh(int A, const PassParams& p, cudaStream_t s);   // packed planes -> fp16 intermediate
bool tc_col_applicable(const PassParams& p, bool any_size);                            // ten strided stages from one plane on the tensor cores
cudaError_t launch_tc_col(const PassParams& p, cudaStream_t s);          // one-plane bits -> fp16 intermediate
cudaError_t tc_timeouts(int* out);
bool tc_row_applicable(const PassParams& p, int T, bool any_size);                     // contiguous 2^14 tiles of the fp16 intermediate, seven or eight stages on the tensor cores
cudaError_t launch_tc_row(int T, const PassParams& p, cudaStream_t s);          // fp16 intermediate -> flip + sum sink
cudaError_t tcrow_timeouts(int* out);
// uplink encoder of a 2^24-long transform as one kernel (strided and contiguous pass side by side)
size_t enc_fused_sync_bytes(int nworkers);                               // zeroed device words the launch needs
cudaError_t launch_enc_fused(const PassParams& pc, const PassParams& pr, int T, int A, uint32_t* sync, cudaStream_t s,
                             bool* launched);
cudaError_t fused_timeouts(int* out);
cudaError_t col_timeouts(int* out);                                      // synchronising read of the strided unit's counter
cudaError_t launch_small(int L, int src, int sink, const PassParams& p, cudaStream_t s);
cudaError_t launch_amplitudes(const void* grads, int bf16, int64_t d, int64_t worker_stride, int M, double alpha,
                              double alpha_s, double n_eff, float* lam, float* lam_s, double* partial, cudaStream_t s);
cudaError_t launch_amplitudes_finalize(const double* partial, int M, int nparts, double alpha, double alpha_s, double n_eff,
                                       float* lam, float* lam_s, cudaStream_t s);
cudaError_t launch_col_norm(int A, const PassParams& p, double* sums, double* room, cudaStream_t s, bool* launched, int* nparts_out);
cudaError_t launch_sum_parts(const double* parts, int64_t nparts, int M, double* sums, int nsums, cudaStream_t s);
// strided pass that also leaves every tile's sum of squares in partial[worker][tile]; *launched stays false where no kernel
// carries them
cudaError_t launch_col_block_norm(int A, int src, const PassParams& p, double* partial, cudaStream_t s, bool* launched, int64_t* parts_per_worker);
// block amplitudes from sums of squares ([M * nb][parts]); lam == nullptr: the server's from finished lam_in alone
cudaError_t launch_block_amplitudes_finalize(const double* seg, int64_t parts, int64_t nb, int M, int block_log2, double alpha,
                                             double alpha_s, float* lam, float* lam_s, cudaStream_t st);
cudaError_t launch_server_amplitudes(const float* lam, int64_t nb, int M, int block_log2, double alpha_s, float* lam_s, cudaStream_t st);
cudaError_t launch_block_amplitudes(const void* grads, int bf16, int64_t d, int64_t dp, int64_t worker_stride, int M,
                                    int block_log2, double alpha, double alpha_s, float* lam, float* lam_s,
                                    double* seg, cudaStream_t st);

}  // namespace fosgd
