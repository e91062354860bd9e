// The decode kernel: attention of one query group over a quantised key cache, or over binary16 keys and values.
//
// Grid (split, KV head x query chunk, sequence).  Every warp prepares the block's (up to 8) query heads as matrix
// fragments in its own registers (ahead of the wait on the preceding kernel), then walks its own 32-key tiles with a
// private online-softmax state (sa_tile_mma.cuh): no block-wide barrier in the main loop.
// The warps' states and then the blocks' partial results are merged with exact power-of-two factors.  For
// sa_decode_step the warp that owns the new token's tile writes the token first.
#pragma once
#include "sa_cache_write.cuh"
#include "sa_common.cuh"
#include "sa_decode_common.cuh"
#include "sa_mma.cuh"
#include "sa_stage.cuh"
#include "sa_tile_mma.cuh"

namespace sa {

// Shared-memory plan of one block: [NW warps x NS stage buffers][mbarriers][R of every warp and query][{R, l} of the block
// for every query]; the block merge's rows and the block's sums re-use the stage buffers once every warp has left its tile
// loop.  {R, l} has a place of its own because l carries the mark of a copy that never came: a copy that was merely late
// may still land in its stage buffer.
template <int D, int FMT, int NW, int NS>
struct MmaSmem {
    using Stage = MmaStage<D, FMT>;
    static constexpr int kMbarOff = NW * NS * Stage::kBytes;
    static constexpr int kRefOff = kMbarOff + ((NW * NS * 8 + 127) & ~127);
    static constexpr int kHeadOff = kRefOff + NW * 8 * 4;
    static constexpr int kBytes = kHeadOff + 8 * 8;
    static constexpr int kInOff = kBytes;                     // WHOLE: the unit's queries, new key and new value (host_in)
    static constexpr int kWholeBytes = kInOff + 10 * D * 2;
    static constexpr int kSumOff = NW * 8 * (D + 2) * 4;      // the block's O, behind the merge rows (within the stage buffers)
    static_assert(kSumOff + 8 * D * 4 <= NW * NS * Stage::kBytes, "merge rows and sums must fit in the stage buffers");
    static_assert(kHeadOff >= NW * NS * Stage::kBytes, "no copy may land on the marks");
    static_assert(NW * NS * Stage::kBytes >= kPlanScratchInts * 4, "the block plan's scratch must fit in the stage buffers");
    static_assert(Stage::kBytes == (FMT == FMT_FP16 ? half_block_bytes_fp16(D) : half_block_bytes(D, format_kb<FMT>(), ScoreMma<D, FMT>::kDense)), "a stage buffer is a verbatim copy of half a page block");
};

// This block's share of the outputs of a cluster (a.cluster blocks, each with the O[D] of its query heads at shared address
// `sums` and their {R, l} HEADS bytes behind that) -> O.  All loads of an output are in flight together; the blocks are
// added in order.
template <int D, int NT, int HEADS>
SA_D void merge_cluster(const DecodeArgs& a, uint32_t sums, float* O) {
    constexpr int kMost = kClusterMost;
    const int C = a.cluster, items = a.gt * (D / 2), per = (items + C - 1) / C, rank = blockIdx.x % C;
    for (int i = rank * per + threadIdx.x; i < min(items, (rank + 1) * per); i += NT) {
        const int g = i / (D / 2), col = i % (D / 2);
        float2 h[kMost], v[kMost];
        int Rm = kMNone;
#pragma unroll
        for (int k = 0; k < kMost; ++k) {
            h[k] = v[k] = make_float2(0.0f, 0.0f);
            if (k < C) {
                const uint32_t row = C > 1 ? cluster_map(sums, k) : sums;
                h[k] = C > 1 ? lds_cluster_f2(row + HEADS + g * 8) : lds_f2(row + HEADS + g * 8);
                v[k] = C > 1 ? lds_cluster_f2(row + (g * D + 2 * col) * 4) : lds_f2(row + (g * D + 2 * col) * 4);
                Rm = max(Rm, __float_as_int(h[k].x));
            }
        }
        float l = 0.0f, x = 0.0f, y = 0.0f;
#pragma unroll
        for (int k = 0; k < kMost; ++k)
            if (k < C) {
                const float f = pow2i_neg(__float_as_int(h[k].x) - Rm);            // (a block without a key carries zeros)
                l += h[k].y * f;
                x += v[k].x * f;
                y += v[k].y * f;
            }
        // no key at all: zeros; a marked sum (a bounded wait gave up) stays visible as NaN
        const float inv = l == 0.0f ? 0.0f : 1.0f / l;
        *reinterpret_cast<float2*>(O + (size_t)g * D + 2 * col) = make_float2(x * inv, y * inv);
    }
}

// The unit's inputs from host memory into every block of the cluster: queries (gt rows), new key, new value at `in`.  The first
// block fetches them (blocks that ask for the same lines of host memory at once are served one after another), while the others
// start; nothing here waits for the preceding kernels, none of which writes host inputs.
template <int D>
SA_D void fetch_inputs(const DecodeArgs& a, uint32_t in, int b, int kvh) {
    const int C = a.cluster, rank = blockIdx.x % C, nq = a.gt * (D / 8), nk = D / 8, i = threadIdx.x;
    uint4 x = make_uint4(0u, 0u, 0u, 0u);
    const bool mine = rank == 0 && i < nq + 2 * nk;
    if (mine) {
        const size_t unit = (size_t)b * a.Hkv + kvh;
        const uint16_t* src = i < nq ? a.Q + unit * a.gt * D + i * 8 : (i < nq + nk ? a.Knew + (i - nq) * 8 : a.Vnew + (i - nq - nk) * 8) + unit * D;
        x = __ldcv(reinterpret_cast<const uint4*>(src));      // host memory: never from a cache line of an earlier step
    }
    if (C > 1) cluster_sync();                                // every block of the cluster is there
    if (mine)
        for (int r = 0; r < C; ++r) sts_cluster_u4(C > 1 ? cluster_map(in + i * 16, r) : in + i * 16, x);
    if (C > 1) cluster_sync();
    else __syncthreads();
}

// CODE: the cache-write mode of the fused append (see write_token).  LOST: the test hook that never issues one chosen
// tile's copy and makes its first plan for another block's coordinates (sa_debug_decode_lost_copy).
// At most 112 registers at d = 64: what two blocks of 256 threads then leave of an SM are two blocks of the merge kernel, which
// stand by while these end (8 x 19 323 tokens, 8 / 2 heads, PoT-4: 14.9 us a call with room for one, 13.9 for two).
// WHOLE: the splits of a sequence form one cluster (or there is one split), which merges them (merge_cluster); an
// instantiation of its own, as the code at the end costs the others 0.1 - 0.3 us.
template <int D, int FMT, int CODE, int NW, int BPS, int NS, bool LOST, bool WHOLE>
__global__ void __maxnreg__(D == 128 ? 168 : 112) decode_mma_kernel(const __grid_constant__ DecodeArgs a) {
    using SM = MmaSmem<D, FMT, NW, NS>;
    using Stage = typename SM::Stage;
    constexpr uint32_t kPolls = LOST ? (1u << 10) : kWaitLimit;
    extern __shared__ __align__(1024) uint8_t smem[];

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int GT = a.gt;                           // query heads of this block (1 .. 8)
    const int chunks = a.G / GT;
    const int kvh = blockIdx.y / chunks;
    const int h0 = kvh * a.G + (blockIdx.y % chunks) * GT;
    // What this block works on: sequence z and split x of the host's n_splits, or (batches of 2 .. 128 sequences) what
    // plan_block deals it from the cached lengths.  The plan made here, from lengths the preceding kernel may be about
    // to change, is a guess that lets the query preparation run ahead of the dependency wait; the plan made after the
    // wait decides, and the preparation is repeated in the rare case that it names another sequence.
    const bool ranked = batch_is_ranked(a.batch) && !(WHOLE && a.cluster > 1);     // (clusters: every sequence has its own)
    int* plan_scratch = reinterpret_cast<int*>(smem);
    BlockPlan bp{(int)blockIdx.z, (int)blockIdx.x, a.n_splits, 0};
    if (a.wait_first) pdl_wait();
    if (ranked)
        bp = plan_block(plan_args(a), LOST ? (blockIdx.z + 1) % a.batch : blockIdx.z, blockIdx.x, false, a.wait_first != 0, bp, plan_scratch);
    const uint32_t mbar0 = smem_addr(smem + SM::kMbarOff) + warp * NS * 8;
    const uint32_t stage0 = smem_addr(smem) + warp * NS * Stage::kBytes;

    if (lane == 0) {
#pragma unroll
        for (int s = 0; s < NS; ++s) mbar_init(mbar0 + s * 8, 1u);
        fence_mbar_init();
        fence_proxy_async();
    }
    __syncwarp();
    pdl_launch_dependents();    // the split-K merge may be scheduled as soon as blocks of this grid retire

    const uint16_t* host_rows = nullptr;
    if constexpr (WHOLE)
        if (a.host_in) {
            fetch_inputs<D>(a, smem_addr(smem + SM::kInOff), blockIdx.z, kvh);
            host_rows = reinterpret_cast<const uint16_t*>(smem + SM::kInOff);
        }
    TileMma<D, FMT, false, false> t;
    int b = bp.b, n_tiles_g, first_g, tile1_g, pidx_g, lp_g, pnew_g;
    bool again;
#pragma unroll 1
    do {
        const int split_g = bp.split, nsp_g = bp.n_splits;         // what the hint below is computed for
        const int bq = b < 0 ? 0 : b;                              // (a block without work so far prepares sequence 0)
        const int len_g = (ranked ? bp.len : __ldcg(a.seq_lens + bq)) + (a.Knew ? 1 : 0);
        // ---- queries: reads only Q, which no kernel of a decode step writes, so it runs before the wait ----
        const uint16_t* q_rows = WHOLE && host_rows ? host_rows : a.Q + ((size_t)bq * a.Hq + h0) * D;
        t.load_queries((lane >> 2) < GT ? q_rows + (lane >> 2) * D : nullptr, lane, a.hadamard != 0, a.zscale);
        // A guess at this warp's first tile, only to ask L2 for it while the preceding kernel drains (loads that bypass
        // L1, so nothing stale can be read back later).
        n_tiles_g = (min(max(len_g, 0), a.max_pages * kPageTokens) + 31) >> 5;
        first_g = split_begin(n_tiles_g, bp.split, bp.n_splits) + warp;
        tile1_g = split_begin(n_tiles_g, bp.split + 1, bp.n_splits);
        lp_g = a.Knew && len_g > 0 ? (len_g - 1) / kPageTokens : -1;          // the new token's page
        if (lp_g >= a.max_pages) lp_g = -1;
        if (first_g < tile1_g) {
            const int p_g = __ldcg(a.page_table + (size_t)bq * a.max_pages + (first_g >> 1));
            if (lane == 0 && p_g >= 0 && p_g < a.n_pages)
                Stage::prefetch(a.pages + ((size_t)p_g * a.Hkv + kvh) * a.page_bytes, (first_g & 1) * 32, true);
        }
        pdl_wait();                 // everything below reads what the preceding kernels in the stream wrote (the cache)
        // The pages of the guessed first tile and of the new token, read again now that they are valid, at the same time as
        // the length(s): one round trip where the guess holds, which it does unless a length crossed a tile boundary.  The
        // warp that is to write the new token asks for its rows as well.
        const int32_t* table_g = a.page_table + (size_t)bq * a.max_pages;
        pidx_g = first_g < tile1_g ? table_g[first_g >> 1] : -1;
        pnew_g = lp_g >= 0 ? table_g[lp_g] : -1;
        if (lp_g >= 0 && !a.host_in && n_tiles_g - 1 >= first_g && n_tiles_g == tile1_g && (n_tiles_g - 1 - first_g) % NW == 0) {
            const size_t row = ((size_t)bq * a.Hkv + kvh) * D;
            asm volatile("prefetch.global.L1 [%0];" ::"l"(a.Knew + row + lane * (D / 32)));
            asm volatile("prefetch.global.L1 [%0];" ::"l"(a.Vnew + row + lane * (D / 32)));
        }
        again = false;
        if (ranked && !a.wait_first) {                            // the plan that counts; wait_first made it after the wait already
            bp = plan_block(plan_args(a), blockIdx.z, blockIdx.x, !LOST, true, bp, plan_scratch);
            again = bp.b != bq && bp.b >= 0;
            if (bp.split != split_g || bp.n_splits != nsp_g) n_tiles_g = -1;  // the guess was for other tiles
            if (bp.b != bq) n_tiles_g = lp_g = -1;
            b = bp.b;
        }
    } while (again);
    if (ranked && b < 0) {                                        // more blocks than (sequence, split) pairs
        if (WHOLE && a.arrivals && warp == 0) bump_lengths(a, lane);
        return;
    }

    // ---- this warp's tiles ----
    int len = ranked ? bp.len : a.seq_lens[b];
    const int32_t* table = a.page_table + (size_t)b * a.max_pages;
    int tile_new = -1, pidx_new = -1;
    if (a.Knew) {
        // Fused append: the step's new token goes to position len (if its page is mapped) and is part of this step's
        // attention.  Every block takes the same decision; the split-K merge kernel bumps seq_lens once all have read it.
        const int lp = len / kPageTokens;
        pidx_new = (len >= 0 && lp < a.max_pages) ? (lp == lp_g ? pnew_g : table[lp]) : -1;
        if (pidx_new >= 0 && pidx_new < a.n_pages) {
            tile_new = len >> 5;
            len += 1;
        }
    }
    const int n_tiles = (min(len, a.max_pages * kPageTokens) + 31) >> 5;
    const bool same = n_tiles == n_tiles_g;                       // the divisions of the guess stand
    const int first = same ? first_g : split_begin(n_tiles, bp.split, bp.n_splits) + warp;
    const int tile1 = same ? tile1_g : split_begin(n_tiles, bp.split + 1, bp.n_splits);
    const int n_my = first < tile1 ? (tile1 - first + NW - 1) / NW : 0;
    // which of my tiles is the new token's (warp-uniform; the others' copies start before the token is encoded)
    const int i_new = (tile_new >= first && tile_new < tile1 && (tile_new - first) % NW == 0) ? (tile_new - first) / NW : -1;
    // Start the copy of a tile of mine, whose page is `pidx`, into the stage buffer at `st` with the mbarrier `mb`; returns how
    // many of its keys count (32 or more: all).  A tile whose page is not mapped gets a plain arrival instead, which completes
    // the phase, and counts for none.
    constexpr bool kEvenStep = NW % 2 == 0;                       // all tiles of a warp are the same half of their pages
    const uint8_t* pool = a.pages + (size_t)kvh * a.page_bytes + (kEvenStep ? (first & 1) * Stage::kBytes : 0);
    const uint32_t page_step = (uint32_t)a.Hkv * (uint32_t)a.page_bytes;      // (the host refuses 2^32 and more)
    auto issue = [&](int tile, int pidx, uint32_t st, uint32_t mb) {
        const bool mapped = (unsigned)pidx < (unsigned)a.n_pages;
        if (lane == 0 && !(LOST && tile == a.lost_tile && b == a.lost_b && kvh == a.lost_kvh)) {     // test hook: that copy never starts
            if (mapped) Stage::issue(st, pool + (uint64_t)(uint32_t)pidx * page_step, kEvenStep ? 0 : (tile & 1) * 32, mb);
            else mbar_arrive(mb);
        }
        return mapped ? len - tile * 32 : 0;
    };
    int n_keys[NS];                                               // of the tiles in flight, the next one first
#pragma unroll
    for (int i = 0; i < NS; ++i)
        if (i < n_my && i != i_new) {
            const int pidx = (same && i == 0) ? pidx_g : table[(first + NW * i) >> 1];
            n_keys[i] = issue(first + NW * i, pidx, stage0 + i * Stage::kBytes, mbar0 + i * 8);
        }
    if (i_new >= 0) {                                             // encode / quantise the token, write it into its page, copy its tile
        CacheArgs ca{};
        ca.page_bytes = a.page_bytes;
        ca.kcode_off = a.kcode_off;
        ca.meta_off = a.meta_off;
        ca.v_off = a.v_off;
        ca.plane_off = a.plane_off;
        ca.hadamard = a.hadamard;
        ca.k = a.k;
        uint8_t* block = const_cast<uint8_t*>(a.pages) + ((size_t)pidx_new * a.Hkv + kvh) * a.page_bytes;
        const size_t row = ((size_t)b * a.Hkv + kvh) * D;
        const bool fetched = WHOLE && host_rows;
        write_token<D, CODE>(block, ca, (len - 1) % kPageTokens, lane, fetched ? host_rows + GT * D : a.Knew + row,
                             fetched ? host_rows + (GT + 1) * D : a.Vnew + row);
        fence_proxy_async_global();
        __syncwarp();
#pragma unroll
        for (int i = 0; i < NS; ++i)
            if (i == i_new) n_keys[i] = issue(tile_new, pidx_new, stage0 + i * Stage::kBytes, mbar0 + i * 8);
    }

    t.start();
    bool failed = false;
    uint32_t st = stage0, mb = mbar0;
    const int32_t* next_page = table + ((first + NW * NS) >> 1);
    int tile = first;
    for (int i = 0; i < n_my; ++i, tile += NW) {
        // the page of the tile that will take this stage over, fetched while this one is worked on
        const int pidx_next = (i + NS < n_my) ? (kEvenStep ? *next_page : table[(tile + NW * NS) >> 1]) : -1;
        next_page += NW / 2;
        // the decision is made warp-uniform: a lane must never leave the loop alone
        const uint32_t parity = (uint32_t)(i / NS) & 1u;
        if (!__all_sync(0xffffffffu, mbar_try_wait(mb, parity)) && !__all_sync(0xffffffffu, mbar_wait_bounded(mb, parity, kPolls))) {
            failed = true;
            // give the other stages' copies (already issued) a bounded chance to land before this warp's buffers are
            // re-used by the block merge
            for (int k = 1; k < NS && i + k < n_my; ++k)
                (void)mbar_wait_bounded(mbar0 + ((i + k) % NS) * 8, (uint32_t)((i + k) / NS) & 1u, kPolls);
            break;
        }
        t.tile(a, st, n_keys[0], lane, b, h0, tile);
        __syncwarp();                                         // every lane is done with this stage
#pragma unroll
        for (int k = 0; k + 1 < NS; ++k) n_keys[k] = n_keys[k + 1];
        if (i + NS < n_my) {
            if (lane == 0) fence_proxy_async();
            n_keys[NS - 1] = issue(tile + NW * NS, pidx_next, st, mb);
        }
        if constexpr (NS == 2) {                              // (addresses of the two stages differ in their sums' halves only)
            st = 2 * stage0 + Stage::kBytes - st;
            mb = 2 * mbar0 + 8 - mb;
        }
    }

    // ---- merge the warps of the block, write the block's partial ----
    static_assert(NS <= 2, "the loop swaps two stages");
    float* ref_s = reinterpret_cast<float*>(smem + SM::kRefOff);                   // [NW][8]
    float (*red_s)[8][D + 2] = reinterpret_cast<float (*)[8][D + 2]>(smem);        // {unused, l, O[D]}
    const bool poisoned = t.template merge_rows<NW>(ref_s, red_s, lane, warp, failed, [&] {
        if (WHOLE && a.arrivals) bump_lengths(a, lane);           // every warp of the block has read the lengths
    });
    __syncthreads();
    const int slot = ranked ? blockIdx.z * a.n_splits + blockIdx.x : blockIdx.x * a.batch + blockIdx.z;
    // the block's {R, l} and O of every head: the partial, or for the merge within the cluster
    float* head_out = WHOLE ? reinterpret_cast<float*>(smem + SM::kHeadOff) : a.partials + ((size_t)slot * a.Hq + h0) * (D + 2);
    float* sum_out = WHOLE ? reinterpret_cast<float*>(smem + SM::kSumOff) : head_out + 2;
    constexpr int kHeadStep = WHOLE ? 2 : D + 2, kSumStep = WHOLE ? D : D + 2;
    sum_rows<D, NW>(ref_s, red_s, GT, poisoned, sum_out, kSumStep, head_out, kHeadStep);
    if constexpr (WHOLE) {
        if (a.cluster > 1) cluster_sync();
        else __syncthreads();
        merge_cluster<D, 32 * NW, SM::kHeadOff - SM::kSumOff>(a, smem_addr(smem + SM::kSumOff), a.O + ((size_t)b * a.Hq + h0) * D);
        if (a.cluster > 1) cluster_sync();                                         // no block may leave while others read its sums
    }
}

template <int D, int FMT, int CODE, int NW, int BPS, int NS, bool LOST, bool WHOLE>
static void launch_mma_as(const DecodeArgs& a, dim3 grid, cudaStream_t s) {
    constexpr int bytes = WHOLE ? MmaSmem<D, FMT, NW, NS>::kWholeBytes : MmaSmem<D, FMT, NW, NS>::kBytes;
    static OncePerDevice once;
    if (!allow_shared(decode_mma_kernel<D, FMT, CODE, NW, BPS, NS, LOST, WHOLE>, bytes, once)) return;      // (the caller asks for the last error)
    (void)launch_pdl_cluster(decode_mma_kernel<D, FMT, CODE, NW, BPS, NS, LOST, WHOLE>, grid, dim3(32 * NW), (size_t)bytes, s,
                             (unsigned)a.cluster, a);
}
template <int D, int FMT, int CODE, int NW, int BPS, int NS>
static void launch_mma(const DecodeArgs& a, dim3 grid, cudaStream_t s) {
    constexpr KernelShape sh = FMT == FMT_FP16 ? KernelShape{NW, BPS, NS} : cluster_shape(D);
    if (a.cluster > 1) launch_mma_as<D, FMT, CODE, sh.warps, sh.blocks_per_sm, sh.stages, false, true>(a, grid, s);
    else if (a.whole) launch_mma_as<D, FMT, CODE, NW, BPS, NS, false, true>(a, grid, s);
    else launch_mma_as<D, FMT, CODE, NW, BPS, NS, false, false>(a, grid, s);
}

}  // namespace sa
