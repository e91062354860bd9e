// The decode kernel: attention of one query group over a quantised key cache, or over binary16 keys and values.
//
// Grid (split, KV head x query chunk, sequence).  Every warp prepares the block's (up to 8) query heads as matrix
// fragments in its own registers (ahead of the wait on the preceding kernel), then walks its own 32-key tiles with a
// private online-softmax state: no block-wide barrier in the main loop.  Per tile, on fragments throughout:
//   scores   exact integer products of the decoded key codes and the queries (sa_score_mma.cuh): keys x queries;
//   softmax  lane (r, c): keys r, r + 8, r + 16, r + 24 of queries 2 c, 2 c + 1.  The weight of a value row is
//            w = 2^(z - g - R) with an integer reference R per query that bounds z - g from above to within two bits
//            (z: logit in the log2 domain, 2^-g: the value's scale); the normaliser sums 2^(z - R).  R moves (and the
//            state is rescaled by the exact power of two) only when a weight would leave the range of binary16;
//   A.V      O^T[dims][queries] += V^T[dims][keys] w[keys][queries] as m16n8k16 products: INT8 values are exact in
//            binary16, every weight enters as the sum of two binary16 terms (22 significant bits for weights within
//            2^-17 of the largest, an absolute 2^-38 of it below), accumulation in FP32.  The weights reach the operand layout
//            through movmatrix, without shared memory.  (Binary16 values: one term, the weights rounded to binary16.)
// The warps' states and then the blocks' partial results are merged with exact power-of-two factors.  For
// sa_decode_step the warp that owns the new token's tile writes the token first.
#pragma once
#include "sa_cache_write.cuh"
#include "sa_common.cuh"
#include "sa_decode_common.cuh"
#include "sa_mma.cuh"
#include "sa_score_mma.cuh"
#include "sa_stage.cuh"

namespace sa {

constexpr int kWeightShift = 14;          // weights are scaled by 2^14: the largest (2^1.98 above R) stays below 65504
// |R| <= 2^28.  R is a float, so from 2^24 on it lies on a grid, of 16 at the limit.  It is rounded up (the reference must not
// lie below z - g by more than the 1.98 that the weights have to spare), which leaves the largest weight at 2^-3 at least:
// 21 bits in two binary16 terms.  A row with a larger logit comes out as NaN; a small integer beside R, right up to
// 1.6e9, cost 0 - 2 % of every call in a loop of its own and 2 - 6 % in the loop of the others.
constexpr float kRefMax = 268435456.0f;

template <int FMT>
constexpr int format_kb() { return FMT == FMT_PLANAR1 ? 1 : FMT == FMT_PLANAR2 ? 2 : FMT == FMT_INT8 ? 8 : 0; }

// Shared-memory plan of one block: [NW warps x NS stage buffers][mbarriers][R of every warp and query][{R, l} of the block
// for every query]; the block merge's rows and the block's sums re-use the stage buffers once every warp has left its tile
// loop.  {R, l} has a place of its own because l carries the mark of a copy that never came: a copy that was merely late
// may still land in its stage buffer.
template <int D, int FMT, int NW, int NS>
struct MmaSmem {
    using SC = ScoreMma<D, FMT>;
    static constexpr int PLANES = FMT == FMT_PLANAR1 ? 1 : FMT == FMT_PLANAR2 ? 2 : 0;
    using Stage = TileStage<SC::CH, FMT != FMT_FP16, FMT == FMT_FP16 ? 2 * D : D, PLANES, D / 8>;
    static constexpr int kMbarOff = NW * NS * Stage::kBytes;
    static constexpr int kRefOff = kMbarOff + ((NW * NS * 8 + 127) & ~127);
    static constexpr int kHeadOff = kRefOff + NW * 8 * 4;
    static constexpr int kBytes = kHeadOff + 8 * 8;
    static constexpr int kSumOff = NW * 8 * (D + 2) * 4;      // the block's O, behind the merge rows (within the stage buffers)
    static_assert(kSumOff + 8 * D * 4 <= NW * NS * Stage::kBytes, "merge rows and sums must fit in the stage buffers");
    static_assert(kHeadOff >= NW * NS * Stage::kBytes, "no copy may land on the marks");
    static_assert(NW * NS * Stage::kBytes >= kPlanScratchInts * 4, "the block plan's scratch must fit in the stage buffers");
    static_assert(Stage::kBytes == (FMT == FMT_FP16 ? half_block_bytes_fp16(D) : half_block_bytes(D, format_kb<FMT>(), SC::kDense)), "a stage buffer is a verbatim copy of half a page block");
};

// The lengths grow by one when the kernel appends the step's tokens and no merge kernel follows: by the hand of the last
// block to get here, every block having read what it needs of them.  One warp per block.
SA_D void bump_lengths(const DecodeArgs& a, int lane) {
    bool last = false;
    if (lane == 0) last = last_to_arrive(a.arrivals, gridDim.x * gridDim.y * gridDim.z);
    if (!__shfl_sync(0xffffffffu, last, 0)) return;
    for (int b = lane; b < a.batch; b += 32) {
        const int len = __ldcg(a.seq_lens + b), lp = len / kPageTokens;
        const int page = (len >= 0 && lp < a.max_pages) ? a.page_table[(size_t)b * a.max_pages + lp] : -1;
        if (page >= 0 && page < a.n_pages) const_cast<int32_t*>(a.seq_lens)[b] = len + 1;
    }
}

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

// CODE: the cache-write mode of the fused append (see write_token).  LOST: the test hook that never issues one chosen
// tile's copy and makes its first plan for another block's coordinates (sa_debug_decode_lost_copy).
// WHOLE: the splits of a sequence form one cluster (or there is one split), which merges them (merge_cluster); an
// instantiation of its own, as the code at the end costs the others 0.1 - 0.3 us.
template <int D, int FMT, int CODE, int NW, int BPS, int NS, bool LOST, bool WHOLE>
__global__ void __launch_bounds__(32 * NW, BPS) decode_mma_kernel(const __grid_constant__ DecodeArgs a) {
    using SM = MmaSmem<D, FMT, NW, NS>;
    using SC = typename SM::SC;
    using Stage = typename SM::Stage;
    constexpr int MT = D / 16;                     // 16-dim row tiles of O^T
    constexpr bool kFp16 = FMT == FMT_FP16;
    constexpr uint32_t kPolls = LOST ? (1u << 10) : kWaitLimit;
    extern __shared__ __align__(1024) uint8_t smem[];

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int r = lane >> 2, c = lane & 3;
    const int GT = a.gt;                           // query heads of this block (1 .. 8)
    const int chunks = a.G / GT;
    const int kvh = blockIdx.y / chunks;
    const int h0 = kvh * a.G + (blockIdx.y % chunks) * GT;
    // What this block works on: sequence z and split x of the host's n_splits, or (batches of 2 .. 128 sequences) what
    // plan_block deals it from the cached lengths.  The plan made here, from lengths the preceding kernel may be about
    // to change, is a guess that lets the query preparation run ahead of the dependency wait; the plan made after the
    // wait decides, and the preparation is repeated in the rare case that it names another sequence.
    const bool ranked = batch_is_ranked(a.batch);
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

    SC q;
    float qs0, qs1;             // logit scale (Delta * log2(e) / sqrt(d) * unit of the scores) of queries 2 c, 2 c + 1
    int b = bp.b, n_tiles_g, first_g, tile1_g, pidx_g, lp_g, pnew_g;
    bool again;
#pragma unroll 1
    do {
        const int split_g = bp.split, nsp_g = bp.n_splits;         // what the hint below is computed for
        const int bq = b < 0 ? 0 : b;                              // (a block without work so far prepares sequence 0)
        const int len_g = (ranked ? bp.len : __ldcg(a.seq_lens + bq)) + (a.Knew ? 1 : 0);
        // ---- queries: reads only Q, which no kernel of a decode step writes, so it runs before the wait ----
        const float qd = q.load(r < GT ? a.Q + ((size_t)bq * a.Hq + h0 + r) * D : nullptr, lane, a.hadamard != 0) * a.zscale;
        qs0 = __shfl_sync(0xffffffffu, qd, 8 * c);
        qs1 = __shfl_sync(0xffffffffu, qd, 8 * c + 4);
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
        if (lp_g >= 0 && n_tiles_g - 1 >= first_g && n_tiles_g == tile1_g && (n_tiles_g - 1 - first_g) % NW == 0) {
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
    // Start the copy of my i-th tile, whose page is `pidx`, into stage i % NS; returns how many of its keys count (32 or more:
    // all).  A tile whose page is not mapped gets a plain arrival instead, which completes the phase, and counts for none.
    const uint8_t* pool = a.pages + (size_t)kvh * a.page_bytes;
    const size_t page_step = (size_t)a.Hkv * a.page_bytes;
    auto issue = [&](int i, int pidx) {
        const int tile = first + NW * i, s = i % NS;
        const bool mapped = pidx >= 0 && pidx < a.n_pages;
        if (lane == 0 && !(LOST && tile == a.lost_tile && b == a.lost_b && kvh == a.lost_kvh)) {     // test hook: that copy never starts
            if (mapped) Stage::issue(stage0 + s * Stage::kBytes, pool + pidx * page_step, (tile & 1) * 32, mbar0 + s * 8);
            else mbar_arrive(mbar0 + s * 8);
        }
        return mapped ? len - tile * 32 : 0;
    };
    int n_keys[NS];                                               // of the tiles in flight, the next one first
#pragma unroll
    for (int i = 0; i < NS; ++i)
        if (i < n_my && i != i_new) {
            const int pidx = (same && i == 0) ? pidx_g : table[(first + NW * i) >> 1];
            n_keys[i] = issue(i, pidx);
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
        write_token<D, CODE>(block, ca, (len - 1) % kPageTokens, lane, a.Knew + row, a.Vnew + row);
        fence_proxy_async_global();
        __syncwarp();
#pragma unroll
        for (int i = 0; i < NS; ++i)
            if (i == i_new) n_keys[i] = issue(i, pidx_new);
    }

    float R0 = 0.0f, R1 = 0.0f;                    // references of queries 2 c, 2 c + 1 (integers)
    bool seen = false;                             // no key yet: R is not set
    f32x2 l = pack_f32x2(0.0f, 0.0f);              // this lane's share of the normalisers
    const f32x2 qs = pack_f32x2(qs0, qs1);
    float acc[MT][4];                              // O^T tiles: dims 16 mt + 2 r (c0, c1), + 1 (c2, c3) of queries 2 c, 2 c + 1
#pragma unroll
    for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[mt][e] = 0.0f;
    bool failed = false;

    for (int i = 0; i < n_my; ++i) {
        const int tile = first + NW * i;
        const int s = i % NS;
        // the page of the tile that will take this stage over, fetched while this one is worked on
        const int pidx_next = (i + NS < n_my) ? table[(tile + NW * NS) >> 1] : -1;
        // the decision is made warp-uniform: a lane must never leave the loop alone
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(mbar0 + s * 8, (uint32_t)(i / NS) & 1u, kPolls))) {
            failed = true;
            // give the other stages' copies (already issued) a bounded chance to land before this warp's buffers are
            // re-used by the block merge
            for (int k = 1; k < NS && i + k < n_my; ++k)
                (void)mbar_wait_bounded(mbar0 + ((i + k) % NS) * 8, (uint32_t)((i + k) / NS) & 1u, kPolls);
            break;
        }
        {
            const uint32_t st = stage0 + s * Stage::kBytes;
            const int n_valid = n_keys[0];

            // ---- scores ----
            float z[4][2], zh[SC::NACC == 2 ? 4 : 1][2];
            q.tile(st, st + Stage::kPlaneOff, lane, a.one, z, zh);
            if (a.dbg_scores) {                               // parity tests only
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int e = 0; e < 2; ++e)
                        if (8 * j + r < n_valid && 2 * c + e < GT) {
                            int A = (int)(z[j][e] * a.score_unit);
                            if constexpr (SC::NACC == 2) A += (int)(zh[j][e] * a.score_unit);
                            a.dbg_scores[((size_t)b * a.Hq + h0 + 2 * c + e) * a.dbg_stride + (size_t)tile * 32 + 8 * j + r] =
                                (int)((uint32_t)A << a.f_extra);
                        }
            }
            // ---- logits and weights ----
            // The lane's two queries as packed FP32: the same arithmetic in half the instructions, and in few enough registers
            // (120 at d = 64) that a block of the merge kernel fits beside two of these: it is then there before the last of
            // them ends.  A step of one sequence of 32 768 tokens took 10.85 us, 9.64 since.
            f32x2 zq[4];                                      // logit per score unit
            float vs[4];                                      // +- 2^(14 - g_j)
            uint32_t meta[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if constexpr (kFp16) {                        // no scales
                    meta[j] = 0u;
                    vs[j] = (float)(1 << kWeightShift);
                    zq[j] = qs;
                } else {
                    meta[j] = lds_u32(st + Stage::kMetaOff + (8 * j + r) * 4);
                    const float sj = half_bits_to_float(meta[j] & 0xffffu);
                    // byte 2 is g_j, in [-10, 30] for written tokens: its place in the exponent field is 7 bits further up, by
                    // a multiplication, for the pipe of the additions.  A negative g_j, 256 too large, toggles the sign bit.
                    vs[j] = __uint_as_float(((127u + kWeightShift) << 23) - (meta[j] & 0x00ff0000u) * 128u);
                    zq[j] = mul2(qs, pack_f32x2(sj, sj));
                }
                if constexpr (SC::NACC == 2) {                // rounded once, like the conversion of one integer sum
                    z[j][0] += zh[j][0];
                    z[j][1] += zh[j][1];
                }
            }
            float p[4][2], w[4][2];
            __half2 h[4];
            bool move = !seen;                                // warp-uniform; rare after the first tile
            for (int turn = 0; turn < 2; ++turn) {            // (a reference that has moved fits)
                if (move) {
                    float y0 = -INFINITY, y1 = -INFINITY;     // largest z - g of the tile, not rounded down
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (8 * j + r < n_valid) {
                            const float g = (float)((int)(meta[j] << 8) >> 24);
                            float zq0, zq1;
                            unpack_f32x2(zq[j], &zq0, &zq1);
                            y0 = fmaxf(y0, __fmaf_ru(z[j][0], zq0, -g));
                            y1 = fmaxf(y1, __fmaf_ru(z[j][1], zq1, -g));
                        }
#pragma unroll
                    for (int o = 4; o < 32; o <<= 1) {
                        y0 = fmaxf(y0, __shfl_xor_sync(0xffffffffu, y0, o));
                        y1 = fmaxf(y1, __shfl_xor_sync(0xffffffffu, y1, o));
                    }
                    y0 = fminf(fmaxf(ceilf(y0), -kRefMax), kRefMax);
                    y1 = fminf(fmaxf(ceilf(y1), -kRefMax), kRefMax);
                    if (seen) {
                        y0 = fmaxf(R0, y0);
                        y1 = fmaxf(R1, y1);
                        const float f0 = pow2i_neg(__float2int_rn(R0 - y0)), f1 = pow2i_neg(__float2int_rn(R1 - y1));
                        l = mul2(l, pack_f32x2(f0, f1));
#pragma unroll
                        for (int mt = 0; mt < MT; ++mt) {
                            acc[mt][0] *= f0;
                            acc[mt][1] *= f1;
                            acc[mt][2] *= f0;
                            acc[mt][3] *= f1;
                        }
                    }
                    R0 = y0;
                    R1 = y1;
                    seen = true;
                }
                const f32x2 nR = pack_f32x2(-R0, -R1);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    float x0, x1;
                    unpack_f32x2(ffma2(pack_f32x2(z[j][0], z[j][1]), zq[j], nR), &x0, &x1);
                    p[j][0] = ex2_approx(x0);
                    p[j][1] = ex2_approx(x1);
                    w[j][0] = p[j][0] * fabsf(vs[j]);
                    w[j][1] = p[j][1] * fabsf(vs[j]);
                }
                if (n_valid < 32) {                           // the sequence's last tile: slots past its end may hold anything
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (8 * j + r >= n_valid) p[j][0] = p[j][1] = w[j][0] = w[j][1] = 0.0f;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) h[j] = __floats2half2_rn(w[j][0], w[j][1]);
                // a weight beyond binary16 has become infinite: 0x7c00, the only value that 0x0400 carries into the sign bit
                const __half2 top = __hmax2(__hmax2(h[0], h[1]), __hmax2(h[2], h[3]));
                move = __any_sync(0xffffffffu, ((*reinterpret_cast<const uint32_t*>(&top) + 0x04000400u) & 0x80008000u) != 0u);
                if (__builtin_expect(!move, 1)) break;
            }
            uint32_t bh[4], bl[4];                            // operand fragments: keys 8 j + 2 c, + 1 of query r
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float2 hf = __half22float2(h[j]);
                bh[j] = movmatrix_trans(*reinterpret_cast<const uint32_t*>(&h[j]));
                if constexpr (kFp16) {
                    // one term; the normaliser sums the same rounded weights, so the result is an exact weighted mean
                    l = add2(l, pack_f32x2(hf.x, hf.y));
                } else {
                    l = add2(l, pack_f32x2(p[j][0], p[j][1]));
                    float x0, x1;                             // what the first term leaves
                    unpack_f32x2(ffma2(pack_f32x2(hf.x, hf.y), pack_f32x2(-1.0f, -1.0f), pack_f32x2(w[j][0], w[j][1])), &x0, &x1);
                    const __half2 lo = __floats2half2_rn(x0, x1);
                    bl[j] = movmatrix_trans(*reinterpret_cast<const uint32_t*>(&lo));
                }
            }
            // ---- A.V: an 8 x 8 block of 16-bit pairs (8 keys x 16 dims of INT8), transposed by ldmatrix: row r of
            // the operand is dim 2 r (bytes 0, 2), row r + 8 dim 2 r + 1 (bytes 1, 3), columns the keys 2 c, 2 c + 1 ----
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                uint32_t x[4];
                if constexpr (kFp16) {                        // binary16 values: chunk 2 mt is rows r (dims 16 mt + r), chunk 2 mt + 1 rows r + 8
                    uint32_t y[4];
                    ldmatrix_x4_trans(x, st + Stage::kVOff + 2 * mt * 512 + lane * 16);
                    ldmatrix_x4_trans(y, st + Stage::kVOff + (2 * mt + 1) * 512 + lane * 16);
                    if (n_valid < 32) {
                        // slots past the end may hold anything (even NaN patterns): their weight is zero, but 0 * NaN is not
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const int key = 8 * j + 2 * c;
                            const uint32_t keep = key >= n_valid ? 0u : key + 1 >= n_valid ? 0x0000ffffu : 0xffffffffu;
                            x[j] &= keep;
                            y[j] &= keep;
                        }
                    }
                    mma_f16_16816(acc[mt], x[0], y[0], x[1], y[1], bh[0], bh[1]);
                    mma_f16_16816(acc[mt], x[2], y[2], x[3], y[3], bh[2], bh[3]);
                    continue;
                }
                ldmatrix_x4_trans(x, st + Stage::kVOff + mt * 512 + lane * 16);
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const uint32_t a0 = int8_to_half2<false>(x[2 * k]), a1 = int8_to_half2<true>(x[2 * k]);
                    const uint32_t a2 = int8_to_half2<false>(x[2 * k + 1]), a3 = int8_to_half2<true>(x[2 * k + 1]);
                    mma_f16_16816(acc[mt], a0, a1, a2, a3, bh[2 * k], bh[2 * k + 1]);
                    mma_f16_16816(acc[mt], a0, a1, a2, a3, bl[2 * k], bl[2 * k + 1]);
                }
            }
        }
        __syncwarp();                                         // every lane is done with this stage
#pragma unroll
        for (int k = 0; k + 1 < NS; ++k) n_keys[k] = n_keys[k + 1];
        if (i + NS < n_my) {
            if (lane == 0) fence_proxy_async();
            n_keys[NS - 1] = issue(i + NS, pidx_next);
        }
    }

    // ---- merge the warps of the block, write the block's partial ----
    // R of every warp and query goes to shared memory; every warp scales its state by the exact 2^(R - Rb), Rb the
    // block's largest, and writes it out; the rows are added in a fixed order.
    float* ref_s = reinterpret_cast<float*>(smem + SM::kRefOff);                   // [NW][8]
    float (*red_s)[8][D + 2] = reinterpret_cast<float (*)[8][D + 2]>(smem);        // {unused, l, O[D]}
    float l0, l1;
    unpack_f32x2(l, &l0, &l1);
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {
        l0 += __shfl_xor_sync(0xffffffffu, l0, o);
        l1 += __shfl_xor_sync(0xffffffffu, l1, o);
    }
    if (r == 0) {
        ref_s[warp * 8 + 2 * c] = seen ? R0 : (float)kMNone;
        ref_s[warp * 8 + 2 * c + 1] = seen ? R1 : (float)kMNone;
    }
    // A warp whose bounded wait for a copy expired makes the block's whole partial a marked one: l = NaN is written
    // below from a register, not through the rows, which alias the stage buffers — a copy that was merely late could
    // still land in them.
    const bool poisoned = __syncthreads_or(failed ? 1 : 0) != 0;
    if (WHOLE && a.arrivals && warp == 0) bump_lengths(a, lane);  // every warp of the block has read the lengths
    float Rb0 = (float)kMNone, Rb1 = (float)kMNone;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        Rb0 = fmaxf(Rb0, ref_s[w * 8 + 2 * c]);
        Rb1 = fmaxf(Rb1, ref_s[w * 8 + 2 * c + 1]);
    }
    const float f0 = seen ? pow2i_neg(__float2int_rn(R0 - Rb0)) : 0.0f, f1 = seen ? pow2i_neg(__float2int_rn(R1 - Rb1)) : 0.0f;
    const float v0 = f0 * (1.0f / (1 << kWeightShift)), v1 = f1 * (1.0f / (1 << kWeightShift));
    if (r == 0) {
        red_s[warp][2 * c][1] = l0 * (kFp16 ? v0 : f0);
        red_s[warp][2 * c + 1][1] = l1 * (kFp16 ? v1 : f1);
    }
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
        if constexpr (kFp16) {
            const int dim = 16 * mt + r;
            red_s[warp][2 * c][2 + dim] = acc[mt][0] * v0;
            red_s[warp][2 * c][2 + dim + 8] = acc[mt][2] * v0;
            red_s[warp][2 * c + 1][2 + dim] = acc[mt][1] * v1;
            red_s[warp][2 * c + 1][2 + dim + 8] = acc[mt][3] * v1;
            continue;
        }
        const int dim = 16 * mt + 2 * r;
        *reinterpret_cast<float2*>(&red_s[warp][2 * c][2 + dim]) = make_float2(acc[mt][0] * v0, acc[mt][2] * v0);
        *reinterpret_cast<float2*>(&red_s[warp][2 * c + 1][2 + dim]) = make_float2(acc[mt][1] * v1, acc[mt][3] * v1);
    }
    __syncthreads();
    const int slot = ranked ? blockIdx.z * a.n_splits + blockIdx.x : blockIdx.x * a.batch + blockIdx.z;
    // the block's {R, l} and O of every head: the partial, or for the merge within the cluster
    float* head_out = WHOLE ? reinterpret_cast<float*>(smem + SM::kHeadOff) : a.partials + ((size_t)slot * a.Hq + h0) * (D + 2);
    float* sum_out = WHOLE ? reinterpret_cast<float*>(smem + SM::kSumOff) : head_out + 2;
    constexpr int kHeadStep = WHOLE ? 2 : D + 2, kSumStep = WHOLE ? D : D + 2;
    for (int idx = threadIdx.x; idx < GT * (D / 2); idx += 32 * NW) {              // two dims of one head
        const int g = idx / (D / 2), col = idx % (D / 2);
        float2 v = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const float2 x = *reinterpret_cast<const float2*>(&red_s[w][g][2 + 2 * col]);
            v.x += x.x;
            v.y += x.y;
        }
        *reinterpret_cast<float2*>(sum_out + g * kSumStep + 2 * col) = v;
    }
    if (threadIdx.x >= 32 * NW - 8 && 8 - (32 * NW - (int)threadIdx.x) < GT) {     // R and l (by the last warp: it has no more dims than the others)
        const int g = 8 - (32 * NW - (int)threadIdx.x);
        float Rm = (float)kMNone, l = 0.0f;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            Rm = fmaxf(Rm, ref_s[w * 8 + g]);
            l += red_s[w][g][1];
        }
        *reinterpret_cast<float2*>(head_out + g * kHeadStep) = poisoned ? make_float2(__int_as_float(0), __int_as_float(0x7fc00000))      // R = 0, l = NaN
                                                                        : make_float2(__int_as_float(__float2int_rn(Rm)), l);
    }
    if constexpr (WHOLE) {
        if (a.cluster > 1) cluster_sync();
        else __syncthreads();
        merge_cluster<D, 32 * NW, SM::kHeadOff - SM::kSumOff>(a, smem_addr(smem + SM::kSumOff), a.O + ((size_t)b * a.Hq + h0) * D);
        if (a.cluster > 1) cluster_sync();                                         // no block may leave while others read its sums
    }
}

template <int D, int FMT, int CODE, int NW, int BPS, int NS, bool LOST, bool WHOLE>
static void launch_mma_as(const DecodeArgs& a, dim3 grid, cudaStream_t s) {
    constexpr int bytes = MmaSmem<D, FMT, NW, NS>::kBytes;
    static OncePerDevice once;
    if (!allow_shared(decode_mma_kernel<D, FMT, CODE, NW, BPS, NS, LOST, WHOLE>, bytes, once)) return;      // (the caller asks for the last error)
    (void)launch_pdl_cluster(decode_mma_kernel<D, FMT, CODE, NW, BPS, NS, LOST, WHOLE>, grid, dim3(32 * NW), (size_t)bytes, s,
                             (unsigned)a.cluster, a);
}
template <int D, int FMT, int CODE, int NW, int BPS, int NS>
static void launch_mma(const DecodeArgs& a, dim3 grid, cudaStream_t s) {
    if (a.whole) launch_mma_as<D, FMT, CODE, NW, BPS, NS, false, true>(a, grid, s);
    else launch_mma_as<D, FMT, CODE, NW, BPS, NS, false, false>(a, grid, s);
}

}  // namespace sa
