// Encoder of blocks of 2^16 in one kernel: a cluster of eight thread blocks holds a whole block of the gradient.
//
// Thread block c of the cluster reads columns [c, c + 1) 2^(T-3) of the eight segments of 2^T coordinates, does the top
// three stages across the segments in registers, and stores row s into the shared memory of thread block s, which goes on
// with the T stages of segment s, the dither and the packing as the contiguous pass does.  The two-kernel form (A = 4,
// T = 12) writes and reads the intermediate in between: 16 x 2^23 336 -> 294 us (bf16 359 -> 310), bound by the
// instructions of the dither (187 us) and by what the barriers leave uncovered.  Measuring the blocks' norms on the way, squares
// and sums in fp64, takes 34 us more (bf16 12); their own pass over the gradients took 92 (82).  2^17 with tiles of 2^14, two thread blocks
// per SM, lost: 328 -> 357 us.
#include "row_kernels.cuh"

namespace fosgd {

__device__ __forceinline__ uint32_t cluster_address(const void* mine, uint32_t rank)
{
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"((uint32_t)__cvta_generic_to_shared(mine)), "r"(rank));
    return remote;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, float4 q)
{
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" :: "r"(addr), "f"(q.x), "f"(q.y), "f"(q.z), "f"(q.w) : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t addr, double q)
{
    asm volatile("st.shared::cluster.f64 [%0], %1;" :: "r"(addr), "d"(q) : "memory");
}

// row s of this thread's four columns: coordinates base + s 2^T + 0 .. 3.  WHOLE: all of them inside the gradient.
template <int T, int SRC, bool WHOLE>
__device__ __forceinline__ void load_rows(const PassParams& p, int n, int64_t base, float (&v)[32])
{
    const int64_t left = p.d - base;
    if constexpr (SRC == SRC_G32) {
        const float* const src = static_cast<const float*>(p.src) + (int64_t)n * p.src_stride + base;
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            const int o = s << T;
            float* const x = v + 4 * s;
            if (WHOLE || o + 4 <= left) {
                const float4 q = load_cs(reinterpret_cast<const float4*>(src + o));
                x[0] = q.x; x[1] = q.y; x[2] = q.z; x[3] = q.w;
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) x[k] = o + k < left ? src[o + k] : 0.f;
            }
        }
    } else {
        const uint16_t* const src = static_cast<const uint16_t*>(p.src) + (int64_t)n * p.src_stride + base;
        uint2 q[8];
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            const int o = s << T;
            if (WHOLE || o + 4 <= left) {
                q[s] = load_cs(reinterpret_cast<const uint2*>(src + o));
            } else {
                uint32_t x[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) x[k] = o + k < left ? src[o + k] : 0u;
                q[s] = make_uint2(x[0] | x[1] << 16, x[2] | x[3] << 16);
            }
        }
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            v[4 * s + 0] = __uint_as_float(q[s].x << 16); v[4 * s + 1] = __uint_as_float(q[s].x & 0xFFFF0000u);
            v[4 * s + 2] = __uint_as_float(q[s].y << 16); v[4 * s + 3] = __uint_as_float(q[s].y & 0xFFFF0000u);
        }
    }
}

template <int T, int SRC>
__global__ void __launch_bounds__(1 << (T - 5), min_blocks<T, SINK_PACK1>()) cluster_encode_kernel(const PassParamsRK p)
{
    using C = RowCfg<T>;
    constexpr int W = 1 << (T - 3);            // columns of a block
    extern __shared__ __align__(16) float smem[];
    uint32_t* const fw = reinterpret_cast<uint32_t*>(smem + C::TILE_WORDS);   // [8][W / 32]
    __shared__ float s_amp;
    __shared__ double s_part[8], wsum[C::NT / 32];
    pdl_trigger();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");     // every block has started (waited for below)

    const int tid = threadIdx.x;
    const uint32_t lane = tid & 31, rank = blockIdx.y;
    const int n = blockIdx.z;
    const uint32_t id = p.id0 + (uint32_t)n;
    const int64_t vec_base = (int64_t)blockIdx.x << (T + 3);
    const int64_t tile_base = vec_base + ((int64_t)rank << T);
    const int64_t i0 = tile_base + deposit<C::LMASK, T>(tid);

    // the flips of the block's columns (from the generator alone)
    if (tid < W / 16) {
        const int s = tid / (W / 128), j = tid % (W / 128);
        reinterpret_cast<uint4*>(fw)[tid] = rng_words(p.rng, id, 0u, (uint32_t)((vec_base + ((int64_t)s << T)) >> 7) + rank * (W / 128) + (uint32_t)j);
    }
    pdl_wait();
    if (tid == 0 && p.amp_out == nullptr) s_amp = amplitude_at(p, n, tile_base);

    float v[32];
    const int column = (int)rank * W + 4 * tid;
    if (vec_base + ((int64_t)8 << T) <= p.d) load_rows<T, SRC, true>(p, n, vec_base + column, v);
    else load_rows<T, SRC, false>(p, n, vec_base + column, v);

    double sum = 0.0;
    if (p.amp_out != nullptr) {       // the vector is a block that sets its own amplitude
        sum = sum_of_squares(v);
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
        if (lane == 0) wsum[tid >> 5] = sum;
    }
    __syncthreads();                  // flips, partial sums
#pragma unroll
    for (int s = 0; s < 8; ++s) {
        const uint32_t w = fw[s * (W / 32) + (tid >> 3)];
        const uint32_t pos = (4u * tid) & 31u;
#pragma unroll
        for (int k = 0; k < 4; ++k) v[4 * s + k] = flip_by_bit(v[4 * s + k], w, pos + k);
    }
    butterflies32<0x1C>(v);
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
#pragma unroll
    for (int s = 0; s < 8; ++s)
        st_cluster(cluster_address(smem, s) + 4u * (uint32_t)column, make_float4(v[4 * s], v[4 * s + 1], v[4 * s + 2], v[4 * s + 3]));
    if (p.amp_out != nullptr && tid < 8) {
        double mine = wsum[0];
        for (int k = 1; k < C::NT / 32; ++k) mine += wsum[k];
        st_cluster(cluster_address(s_part + rank, (uint32_t)tid), mine);
    }
    cluster_sync();                   // the block's segment is complete; nobody writes to another block from here on

    if (tid == 0 && p.amp_out != nullptr) {
        sum = s_part[0];
        for (int k = 1; k < 8; ++k) sum += s_part[k];
        s_amp = fmaxf((float)(p.amp_factor * sqrt(sum)), kMinBlockAmplitude);
        if (rank == 0) p.amp_out[(int64_t)n * p.amp_stride + blockIdx.x] = s_amp;
    }
    const int baseF = deposit<C::FMASK, T>(tid);
    static_assert(C::VB == 2, "groups of four coordinates");
#pragma unroll
    for (int g = 0; g < 8; ++g) {
        const float* const q = smem + (baseF | round_F_offset<T>(g));
        const float4 x = *reinterpret_cast<const float4*>(q);
        v[4 * g] = x.x; v[4 * g + 1] = x.y; v[4 * g + 2] = x.z; v[4 * g + 3] = x.w;
    }
    butterflies32<31>(v);
    __syncthreads();                  // the linear tile has been read: the exchange layout takes its place
    store_round_F<T>(smem, baseF, v);
    __syncthreads();
    round_M<T>(smem, deposit<C::MMASK, T>(tid), v);
    load_round_L(smem, deposit<C::LMASK, T>(tid), v);
    butterflies32<C::ACT_L>(v);
    sink_pack1(p, n, id, i0, lane, v, s_amp);
}

// From eight blocks of 2^16 per worker on: fewer are a chain of short kernels, where the two-kernel form is as fast.  The
// choice, and with it the rounding of the sums, depends on the vector alone, never on the number of workers.
bool cluster_encode_applicable(int L, int64_t dp) { return L == 16 && dp >= (int64_t)1 << 19; }

cudaError_t launch_cluster_encode(int src, const PassParams& p, cudaStream_t s)
{
    using C = RowCfg<13>;
    const dim3 grid((unsigned)(p.dp >> 16), 8, (unsigned)p.nworkers);
    return src == SRC_G16 ? launch<cluster_encode_kernel<13, SRC_G16>>(grid, C::NT, C::SMEM_BYTES, s, 8, with_round_keys(p))
                          : launch<cluster_encode_kernel<13, SRC_G32>>(grid, C::NT, C::SMEM_BYTES, s, 8, with_round_keys(p));
}

}  // namespace fosgd
