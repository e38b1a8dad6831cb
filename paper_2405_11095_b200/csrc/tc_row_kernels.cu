// Contiguous pass of a decoder (14 stages on tiles of 2^14 coordinates, flip, sum over the workers)
// with seven of the stages on the tensor cores (tcgen05, sm_100a).
//
// The source is the fp16 intermediate of the strided pass: integers of magnitude <= 1024.  A tile
// of 2^14 consecutive coordinates is read as a matrix X of 128 rows (index bits 7..13) x 128 columns
// (bits 0..6).  By the recursion H_k = H_1 (x) H_{k-1}, H_{2^14} = H_128 (x) H_4 (x) H_32:
//   1. H_4 over column bits 5, 6 runs in packed fp16 on the plain ALUs while the tile is staged
//      (values <= 4096: still exact in fp16);
//   2. H_128 over the row bits is one 128 x 128 x 128 product D = H_128 Z per tile and worker:
//      A = H_128 as fp16 in tensor memory, B = Z as staged in shared memory (columns contiguous, i.e.
//      MN-major), fp32 accumulators in tensor memory (exact: |D| <= 2^19), eight tcgen05.mma of K = 16
//      issued by one thread, completion through mbarriers;
//   3. H_32 over column bits 0..4 runs in fp32 registers: tcgen05.ld hands every thread 32
//      consecutive columns of one row, which is also one word of the flip vector, so the flip and
//      the sum over the workers follow in the same registers.
// HALVES = 2: the 15 stages of a 2^25 transform.  The top one pairs tiles of 2^14; the two products of a pair, the second
// one added or subtracted, go into one accumulator (fp32, |D| <= 2^20), so every block stages both halves.
// All values are integers below 2^24 in magnitude, so the result equals the plain-ALU kernel's bit
// for bit.
//
// A block keeps a tile position and walks the workers (sums in registers), then moves to its next tile.  Its
// warps are specialised, so that nobody waits for two things in turn: a load warp keeps whole tiles (32 KiB, contiguous)
// arriving through the bulk copy engine into a ring of three landing slots; four staging warps turn landed tiles
// into the operand layout in one of two operand buffers; one warp issues the products into three accumulators in
// turn; one warp makes the flip words; sixteen drain warps take the accumulators through the register stages.
// (With sixteen warps that staged an item and then drained the one before, an item took 1.6 us, twice what its 350
// instructions per warp or its shared-memory traffic cost.)  Synchronisation is by mbarriers only (slot landed / read,
// operand full / free, accumulator full / free, flips ready); every wait is bounded.
//
// 2^24 x 32: 0.305 ms (0.357 with warps that staged and drained in turn, 0.324 before the operand was 128-byte swizzled
// and the ring positions 32-bit), 2^25 x 8 0.265.  Bound by the staging warps' chain (without product and drain the rest
// alone takes 0.225 ms) and the shared-memory port; eight staging warps, four accumulators or ring slots, and flips
// made by the staging warps all measured slower or the same.
#include "tc_common.cuh"

namespace fosgd {

static __device__ int g_tcrow_wait_timeouts;   // warps that abandoned a bounded wait

namespace {

constexpr int kT = 14;
constexpr int kDrainWarps = 16, kStageWarps = 4;
constexpr int kFirstStageWarp = kDrainWarps, kIssueWarp = kDrainWarps + kStageWarps, kLoadWarp = kIssueWarp + 1, kFlipWarp = kIssueWarp + 2;
constexpr int kThreads = (kFlipWarp + 1) * 32;             // 736: 80 registers each
constexpr int kAcc = 3;                                    // accumulators (128 columns of tensor memory each) and flip buffers in turn
constexpr int kRing = 3;                                   // landing slots for whole tiles (bulk copies in flight)
constexpr uint32_t kTileBytes = 2u << kT;                  // one fp16 tile
constexpr uint32_t kAColumns = 64;                         // H_128 as fp16 in tensor memory: lane = row, two k per 32-bit column
constexpr uint32_t kTmemColumns = 512;                     // kAcc accumulators of 128 columns, then H_128
constexpr uint32_t kOffB = 0;                              // two operand buffers
constexpr uint32_t kBBlock = 128 * 128;                    // 64 columns x 128 rows k of an operand buffer
constexpr uint32_t kBBytes = 2 * kBBlock;
constexpr uint32_t kOffFlips = kOffB + 2 * kBBytes;        // kAcc buffers of 128 rows x 4 flip words
constexpr uint32_t kOffLand = kOffFlips + kAcc * 2048;     // kRing landing slots
constexpr uint32_t kOffBar = kOffLand + kRing * kTileBytes;   // mbarriers, stop word, tensor-memory base
constexpr int kNumBars = 4 + 3 * kAcc + 2 * kRing;
constexpr uint32_t kSmemBytes = kOffBar + kNumBars * 8 + 16;

enum { BAR_B_FULL = 0, BAR_B_FREE = 2, BAR_ACC_FULL = 4, BAR_ACC_FREE = 4 + kAcc, BAR_FLIPS = 4 + 2 * kAcc, BAR_LAND_FULL = 4 + 3 * kAcc,
       BAR_LAND_FREE = BAR_LAND_FULL + kRing };

// instruction descriptor: D = f32 (1 << 4), A = B = fp16 (0), A K-major, B MN-major (1 << 16), N = 128, M = 128
constexpr uint32_t kIdescF16 = (1u << 4) | (1u << 16) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
constexpr uint32_t kNegateB = 1u << 14;   // D -= A B

// A from tensor memory
__device__ __forceinline__ void umma_f16(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}

// x with its sign flipped iff the top bit of w is set
__device__ __forceinline__ float flip_top(float x, uint32_t w)
{
    return __uint_as_float(__float_as_uint(x) ^ (w & 0x80000000u));
}

__device__ __forceinline__ void hbutterfly(uint4& a, uint4& b)
{
    __half2* const pa = reinterpret_cast<__half2*>(&a);
    __half2* const pb = reinterpret_cast<__half2*>(&b);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const __half2 x = pa[k], y = pb[k];
        pa[k] = __hadd2(x, y);
        pb[k] = __hsub2(x, y);
    }
}

}  // namespace

template <int HALVES>
__global__ void __launch_bounds__(kThreads, 1) tc_row_final_kernel(const PassParams p, const int ntiles)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    pdl_trigger();
    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const uint32_t lane = tid & 31;
    uint64_t* const bar = reinterpret_cast<uint64_t*>(smem + kOffBar);
    volatile int* const s_stop = reinterpret_cast<volatile int*>(smem + kOffBar + kNumBars * 8);
    uint32_t* const tmem_slot = reinterpret_cast<uint32_t*>(smem + kOffBar + kNumBars * 8 + 4);

    // ---- once per block: the constant operand, barriers, tensor memory ----
    if (warp == kIssueWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kTmemColumns) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar + BAR_B_FULL + b, kStageWarps);
            mbar_init(bar + BAR_B_FREE + b, 1);
        }
#pragma unroll
        for (int b = 0; b < kAcc; ++b) {
            mbar_init(bar + BAR_ACC_FULL + b, 1);
            mbar_init(bar + BAR_ACC_FREE + b, kDrainWarps);
            mbar_init(bar + BAR_FLIPS + b, 1);
        }
#pragma unroll
        for (int r = 0; r < kRing; ++r) {
            mbar_init(bar + BAR_LAND_FULL + r, 1);
            mbar_init(bar + BAR_LAND_FREE + r, kStageWarps);
        }
        *s_stop = 0;
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    const uint32_t tmem_a = tmem_base + kAcc * 128u;
    if (warp < 4) {
        // A[m][k] = (-1)^popcount(m & k): a warp writes the 32 rows of its lane quarter, 16 columns at a time
        const uint32_t m = (uint32_t)tid;
#pragma unroll 1
        for (uint32_t c0 = 0; c0 < kAColumns; c0 += 16) {
            uint32_t w[16];
#pragma unroll
            for (uint32_t c = 0; c < 16; ++c) {
                const uint32_t k = 2u * (c0 + c);
                const uint32_t lo = (__popc(m & k) & 1) ? 0xBC00u : 0x3C00u;
                w[c] = lo | ((lo ^ ((m & 1u) << 15)) << 16);      // k + 1 differs from k in bit 0 alone
            }
            asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
                         ::"r"(tmem_a + (((uint32_t)warp * 32u) << 16) + c0), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]),
                           "r"(w[6]), "r"(w[7]), "r"(w[8]), "r"(w[9]), "r"(w[10]), "r"(w[11]), "r"(w[12]), "r"(w[13]), "r"(w[14]), "r"(w[15]) : "memory");
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    pdl_wait();                     // (the set-up above needs nothing from the kernel before)
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();

    // the blocks of a cluster (gridDim.y of them) take a tile's workers in turn; one block, all of them
    const int n_first = (int)blockIdx.y, n_step = (int)gridDim.y;
    const int W = (p.nworkers - n_first + n_step - 1) / n_step;      // workers of this block
    const int n_end = n_first + W * n_step;
    const int my_tiles = ((int)blockIdx.x < ntiles) ? (ntiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
    const int nitems = my_tiles * W;                // item g: this block's tile number g / W, its worker number g % W

    // where an item sits: first coordinate of its tile and its worker; advanced item by item (worker fastest)
    struct Cursor {
        int64_t tile_base;
        int n;
    };
    const int64_t tile_step = (int64_t)gridDim.x << kT;
    auto advance = [&](Cursor& c) {
        c.n += n_step;
        if (c.n == n_end) {
            c.n = n_first;
            c.tile_base += tile_step;
        }
    };
    const Cursor c_first{(int64_t)blockIdx.x << kT, n_first};
    constexpr auto swizzled = [](uint32_t e) -> uint32_t { return (e & ~31u) | ((((e >> 2) ^ (e >> 7)) & 7u) << 2); };   // split sums: e's group of four

    if (warp == kIssueWarp) {
        // ================= the warp that issues the products =================
        if (lane == 0) {
            bool ok = true;
            int g = 0;
            int tile = (int)blockIdx.x, w = 0;
            RingPos<kAcc> acc;
            RingPos<2> op;
            for (; g < nitems; ++g, acc.next()) {
                const uint32_t b = acc.i;
#pragma unroll
                for (int h = 0; h < HALVES && ok; ++h, op.next()) {
                    const uint32_t sb = op.i;
                    ok = mbar_wait_or_stop(bar + BAR_B_FULL + sb, op.full, s_stop);                          // operand staged
                    if (ok && h == 0) ok = mbar_wait_or_stop(bar + BAR_ACC_FREE + b, acc.free(), s_stop);    // accumulator drained
                    if (!ok) break;
                    tc_fence_after_sync();
                    const uint64_t bdesc = umma_desc_mn128(smem_u32(smem + kOffB + sb * kBBytes), kBBlock, 1024u);
                    // the pair's second half enters its first tile with a plus, its second tile with a minus
                    const uint32_t idesc = (h == 1 && (tile & 1)) ? kIdescF16 | kNegateB : kIdescF16;
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks)   // K = 16 per instruction: eight columns of A, two groups of eight rows of B
                        umma_f16(tmem_base + b * 128u, tmem_a + 8u * ks, bdesc + (uint64_t)(ks * (2048 >> 4)), idesc, h + ks > 0 ? 1u : 0u);
                    umma_commit(bar + BAR_B_FREE + sb);
                }
                if (!ok) break;
                umma_commit(bar + BAR_ACC_FULL + b);
                if (++w == W) {
                    w = 0;
                    tile += (int)gridDim.x;
                }
            }
            if (!ok) {
                if (atomicExch((int*)s_stop, 1) == 0) atomicAdd(&g_tcrow_wait_timeouts, 1);
                // products already committed may still be running: one more bounded wait each before the tensor memory goes back
                for (int h = (g >= kAcc ? g - kAcc : 0); h < g; ++h) mbar_wait(bar + BAR_ACC_FULL + (h % kAcc), (uint32_t)(h / kAcc) & 1u);
                if (HALVES > 1) {   // (the first half of the item given up on)
                    umma_commit(bar + BAR_ACC_FULL + (g % kAcc));
                    mbar_wait(bar + BAR_ACC_FULL + (g % kAcc), (uint32_t)(g / kAcc) & 1u);
                }
            }
        }
    } else if (warp == kLoadWarp) {
        // ================= tiles in through the copy engine =================
        if (lane == 0) {
            Cursor c = c_first;
            bool ok = true;
            int g = 0;        // copies started
            const int nloads = HALVES * nitems;
            RingPos<kRing> slot;
            for (; g < nloads; ++g, slot.next()) {
                const uint32_t r = slot.i;
                if (!mbar_wait_or_stop(bar + BAR_LAND_FREE + r, slot.free(), s_stop)) {   // every staging warp has read the slot
                    ok = false;
                    break;
                }
                const __half* src = static_cast<const __half*>(p.src) + (int64_t)c.n * p.src_stride + c.tile_base;
                if (HALVES == 2) src += (int64_t)((int)(g & 1) - (int)((c.tile_base >> kT) & 1)) * (1 << kT);   // the pair's halves in turn
                if (HALVES == 1 || (g & 1)) advance(c);
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar + BAR_LAND_FULL + r)), "r"(kTileBytes) : "memory");
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                             ::"r"(smem_u32(smem + kOffLand + r * kTileBytes)), "l"(src), "r"(kTileBytes), "r"(smem_u32(bar + BAR_LAND_FULL + r)) : "memory");
            }
            if (!ok && atomicExch((int*)s_stop, 1) == 0) atomicAdd(&g_tcrow_wait_timeouts, 1);
            // copies started but possibly not landed yet: one more bounded wait each, so that the engine is not
            // left writing into shared memory that the next block of this SM may own
            for (int h = (g >= kRing ? g - kRing : 0); h < g; ++h)
                mbar_wait(bar + BAR_LAND_FULL + (h % kRing), (uint32_t)(h / kRing) & 1u);
        }
    } else if (warp == kFlipWarp) {
        // ================= flip words: four generator calls per lane and item, 128 rows x 128 flips =================
        Cursor c = c_first;
        bool ok = true;
        RingPos<kAcc> acc;
        for (int g = 0; g < nitems; ++g, acc.next()) {
            const uint32_t b = acc.i;
            // the drain of item g - kAcc has read its flip words (every warp reads them before it frees the accumulator)
            ok = mbar_wait_or_stop(bar + BAR_ACC_FREE + b, acc.free(), s_stop);
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) break;
            const uint32_t id = p.id0 + (uint32_t)c.n, c0 = (uint32_t)(c.tile_base >> 7);
            advance(c);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t row = lane + 32u * k;
                const uint4 w = rng_words(p.rng, id, 0u, c0 + row);
                uint32_t* const f = reinterpret_cast<uint32_t*>(smem + kOffFlips + b * 2048u) + row;   // word q of row r at 128 q + r
                f[0] = w.x; f[128] = w.y; f[256] = w.z; f[384] = w.w;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(bar + BAR_FLIPS + b);
        }
        if (!ok && lane == 0 && atomicExch((int*)s_stop, 1) == 0) atomicAdd(&g_tcrow_wait_timeouts, 1);
    } else if (warp >= kFirstStageWarp && warp < kIssueWarp) {
        // ================= staging: landed tile -> H_4 over column bits 5, 6 -> operand buffer =================
        const uint32_t st = (uint32_t)tid - kFirstStageWarp * 32u, sq = st & 3u;     // column chunks sq + 4 t of rows row0 + 8 kStageWarps i
        // The eight lanes of a 128-bit access have rows k and k + 4.  Reading, the two rows start 256 bytes multiples apart: the
        // second one reads its chunks with column bit 5 swapped, so that together they cover all banks (its differences
        // come out negated).  Writing, the operand's swizzle keeps the two apart.
        const uint32_t odd = (st >> 2) & 1u, row0 = ((st >> 5) << 3) | (odd << 2) | ((st >> 3) & 3u), negate = odd ? 0x80008000u : 0u;
        const int nloads = HALVES * nitems;
        bool ok = true;
        RingPos<kRing> slot;
        RingPos<2> op;
        for (int g = 0; g < nloads; ++g, slot.next(), op.next()) {
            const uint32_t b = op.i, r = slot.i;
            ok = mbar_wait_or_stop(bar + BAR_LAND_FULL + r, slot.full, s_stop);                            // the tile has landed
            if (ok) ok = mbar_wait_or_stop(bar + BAR_B_FREE + b, op.free(), s_stop);                       // product g - 2 has read the buffer
            if (!ok) break;
#pragma unroll
            for (int i = 0; i < 16 / kStageWarps; ++i) {
                const uint32_t srow = row0 + 8u * kStageWarps * i;
                uint4 pre[4];
                const unsigned char* const land = smem + kOffLand + r * kTileBytes + srow * 256u + sq * 16u;
#pragma unroll
                for (int t = 0; t < 4; ++t) pre[t] = *reinterpret_cast<const uint4*>(land + 64u * ((uint32_t)t ^ odd));
                hbutterfly(pre[0], pre[1]);   // column bit 5
                hbutterfly(pre[2], pre[3]);
                pre[1] = make_uint4(pre[1].x ^ negate, pre[1].y ^ negate, pre[1].z ^ negate, pre[1].w ^ negate);
                pre[3] = make_uint4(pre[3].x ^ negate, pre[3].y ^ negate, pre[3].z ^ negate, pre[3].w ^ negate);
                hbutterfly(pre[0], pre[2]);   // column bit 6
                hbutterfly(pre[1], pre[3]);
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    *reinterpret_cast<uint4*>(smem + kOffB + b * kBBytes + (t >> 1) * kBBlock + swizzled_row_chunk(srow, sq + 4u * (t & 1))) = pre[t];
            }
            // One fence for both proxies' next accesses: the product reads the operand, the copy engine rewrites the slot.
            // (The slot is given back only here: freed right after the loads were issued, without a fence, it was
            // now and then refilled before the last of them had read it.)
            fence_generic_before_async();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(bar + BAR_LAND_FREE + r);
                mbar_arrive(bar + BAR_B_FULL + b);
            }
        }
        if (!ok && lane == 0 && atomicExch((int*)s_stop, 1) == 0) atomicAdd(&g_tcrow_wait_timeouts, 1);
    } else if (warp < kDrainWarps) {
        // ================= drain warps: register stages, flip, sum =================
        const uint32_t lq = (uint32_t)warp & 3u, cw = (uint32_t)warp >> 2;       // lane quarter, 32 of the 128 columns
        const uint32_t jrow = lq * 32u + lane;                                  // output row (index bits 7..13)
        float accv[32];
        bool ok = true;
        Cursor c_drain = c_first;

        // drain item g: accumulator -> registers, H_32 over the 32 columns, flip, add
        RingPos<kAcc> acc;
        auto drain_item = [&]() -> bool {
            const uint32_t b = acc.i;
            const int n = c_drain.n;
            const int64_t tile_base = c_drain.tile_base;
            advance(c_drain);
            if (!mbar_wait_or_stop(bar + BAR_ACC_FULL + b, acc.full, s_stop)) return false;
            tc_fence_after_sync();
            if (!mbar_wait_or_stop(bar + BAR_FLIPS + b, acc.full, s_stop)) return false;
            const uint32_t fw = reinterpret_cast<const uint32_t*>(smem + kOffFlips + b * 2048u)[cw * 128u + jrow];
            const float wamp = (p.amp_mode == AMP_WEIGHT) ? amplitude_at(p, n, tile_base) : 1.f;
            uint32_t raw[32];
            tmem_load32(tmem_base + ((lq * 32u) << 16) + b * 128u + cw * 32u, raw);
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar + BAR_ACC_FREE + b);
            float v[32];
#pragma unroll
            for (int r = 0; r < 32; ++r) v[r] = __uint_as_float(raw[r]);
            butterflies32<31>(v);
            if (p.amp_mode == AMP_WEIGHT) {
#pragma unroll
                for (int r = 0; r < 32; ++r) accv[r] = fmaf(flip_top(v[r], fw << (31 - r)), wamp, accv[r]);
            } else {
#pragma unroll
                for (int r = 0; r < 32; ++r) accv[r] += flip_top(v[r], fw << (31 - r));
            }
            if (n + n_step == n_end && n_step == 1) {
                // the tile's sum is complete: scale and store 32 consecutive coordinates
                const int64_t i0 = tile_base + jrow * 128u + cw * 32u;
                const float sc = p.scale * (p.amp_mode == AMP_SCALE ? amplitude_at(p, 0, tile_base) : 1.f);
                float* const dst = static_cast<float*>(p.dst) + i0;
                if (i0 + 32 <= p.d_out) {
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        store_final4(dst + 4 * q, make_float4(accv[4 * q], accv[4 * q + 1], accv[4 * q + 2], accv[4 * q + 3]), sc, p.overwrite);
                } else {
#pragma unroll
                    for (int r = 0; r < 32; ++r)
                        if (i0 + r < p.d_out) store_final(dst + r, accv[r], sc, p.overwrite);
                }
#pragma unroll
                for (int r = 0; r < 32; ++r) accv[r] = 0.f;
            }
            return true;
        };

#pragma unroll
        for (int r = 0; r < 32; ++r) accv[r] = 0.f;
        for (int g = 0; g < nitems && ok; ++g, acc.next()) ok = drain_item();
        if (!ok && lane == 0 && atomicExch((int*)s_stop, 1) == 0) atomicAdd(&g_tcrow_wait_timeouts, 1);
        if (n_step > 1) {
            // This block's share of the sums into the landing slots: every copy has landed and been read (the last
            // accumulator followed the staging of the last tile; after a wait that gave up the sums are incomplete anyway).  Groups of four are permuted by the row: a warp
            // writes 32 rows 512 bytes apart.
            float* const sums = reinterpret_cast<float*>(smem + kOffLand);
#pragma unroll
            for (int q = 0; q < 8; ++q)
                *reinterpret_cast<float4*>(sums + swizzled(jrow * 128u + cw * 32u + 4u * q)) =
                    make_float4(accv[4 * q], accv[4 * q + 1], accv[4 * q + 2], accv[4 * q + 3]);
        }
    }
    if (n_step > 1) {
        __syncthreads();
        const int64_t tile_base = (int64_t)blockIdx.x << kT;
        cluster_reduce_store<kT>(p, tile_base, reinterpret_cast<const float*>(smem + kOffLand), blockIdx.y, gridDim.y,
                                 p.scale * (p.amp_mode == AMP_SCALE ? amplitude_at(p, 0, tile_base) : 1.f), swizzled);
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == kIssueWarp) {
        __syncwarp();
        tc_fence_after_sync();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemColumns) : "memory");
    }
}

// One packed plane's fp16 intermediate in contiguous tiles of 2^14, and at least three workers to sum: with one or
// two (a single decoder, the downlink) the plain-ALU pass is the faster one (0.033 against 0.041 ms on one vector
// of 2^24, 0.051 against 0.057 on two; 0.069 against 0.068 on three, 0.156 against 0.101 on eight).  The 15 stages of a
// 2^25 transform: from five workers on, whose sums repay staging every tile twice (eight: 0.27 against 0.35 ms).
bool tc_row_applicable(const PassParams& p, int T, bool any_size)
{
    if (p.P != 1 || (p.dp >> kT) < 1 || (p.dp >> kT) > 0x7FFFFFFF) return false;
    return T == kT ? any_size || p.nworkers >= 3 : T == kT + 1 && p.nworkers > 4;
}

cudaError_t launch_tc_row(int T, const PassParams& p, cudaStream_t s)
{
    int sms = 0;
    const cudaError_t e = sm_count(&sms);
    if (e != cudaSuccess) return e;
    const int64_t ntiles = p.dp >> kT;
    // fewer tiles than half the SMs (transforms up to 2^20): clusters of blocks share a tile's workers, one tile each
    const unsigned split = worker_split(ntiles, p.nworkers, sms);
    const dim3 grid((unsigned)(ntiles < sms ? ntiles : sms), split);
    if (T == kT) return launch<tc_row_final_kernel<1>>(grid, kThreads, kSmemBytes, s, split, p, (int)ntiles);
    return launch<tc_row_final_kernel<2>>(grid, kThreads, kSmemBytes, s, split, p, (int)ntiles);
}

cudaError_t tcrow_timeouts(int* out) { return cudaMemcpyFromSymbol(out, g_tcrow_wait_timeouts, sizeof(int)); }

}  // namespace fosgd
