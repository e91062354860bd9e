// The decode kernel for calls with work for every SM: one block per SM, which takes a contiguous stretch of the call's tiles.
//
// The tiles of all (query group, sequence) units follow one another, group by group, and are cut into gridDim.x stretches of
// the same length, whatever the lengths of the sequences are (equal short units into even parts, or not at all: cut_stretch); a
// block works through the units of its stretch one after another.  A unit that lies within one block is finished there; of the others every block leaves a partial, and the last one
// to do so merges them: one launch.  Next to the kernel of sa_decode_mma.cuh, whose blocks each work on one unit, several of them to an SM:
//   * no last wave and no idle SM, whatever the shape;
//   * one prologue and one block merge per SM and unit boundary instead of one per block (about 925 warp instructions for
//     every warp, as much as two tiles);
//   * a warp goes on to the next unit, its copies ahead of it, without waiting for the others;
//   * the warps of an SM end together.  Of two blocks on an SM the scheduler prefers the older one's warps: they ended after
//     18 and 24 us (32 and 40 us in longer calls), and for the rest of the time half of the warps were left.
// Measured with both kernels, us a call: see stream_pays() in sa_host.cu.
//
// Each warp works out the stretch for itself from the sequence lengths (no block barrier), ahead of the wait on the preceding
// kernels from lengths that these may still change, and again behind it if they did.
#pragma once
#include "sa_cache_write.cuh"
#include "sa_common.cuh"
#include "sa_decode_common.cuh"
#include "sa_mma.cuh"
#include "sa_stage.cuh"
#include "sa_tile_mma.cuh"

namespace sa {

// [NW warps x NS stage buffers][mbarriers][lengths of the sequences][factors of every warp and query][R, l of every warp and
// query, twice][rows: O of every warp and query].  The rows have a place of their own, so that a warp goes on to the next unit
// without waiting for the others, where that fits (kApart: for as many heads as there are); the last unit's rows, and all
// where it does not fit, re-use the stage buffers.
template <int D, int FMT, int NW, int NS>
struct StreamSmem {
    using Stage = MmaStage<D, FMT>;
    static constexpr int kMbarOff = NW * NS * Stage::kBytes;
    static constexpr int kLenOff = kMbarOff + ((NW * NS * 8 + 127) & ~127);
    static constexpr int kFactorOff = kLenOff + kRankedBatchMax * 4;
    static constexpr int kHeadOff = kFactorOff + 2 * NW * 8 * 4;
    static constexpr int kRowOff = kHeadOff + 2 * NW * 8 * 8;
    __host__ __device__ static constexpr int row_bytes(int heads) { return NW * heads * TileMma<D, FMT, true, false>::kRowStep * 4; }
    __host__ __device__ static constexpr bool apart(int heads) { return kRowOff + row_bytes(heads) <= 227 * 1024; }
    static constexpr int bytes(int heads) { return kRowOff + (apart(heads) ? row_bytes(heads) : 0); }
    static_assert(row_bytes(8) <= NW * NS * Stage::kBytes, "the rows must fit in the stage buffers");
    static_assert(NW % 2 == 0, "all tiles of a warp are the same half of their pages");
    static_assert(NS <= 2, "the loop swaps two stages");
};

constexpr int kLaneSeqs = kRankedBatchMax / 32;       // sequences per lane, at most
struct Stretch {
    int t0, t1;                   // the block's stretch of all (virtual) tiles
    int each, more, grain;        // stretches are `each` tiles long, the first `more` of them `grain` longer
    int y, b, len, start, tiles;  // its first unit: query group, sequence, length before the call, first virtual tile, real tiles
    int free;                     // virtual tiles in front of the real ones of every unit
};
// Tiles of a sequence of `len` tokens in the cut: an empty one counts as one, so that a block takes care of its output.
SA_D int stretch_tiles(int len, int cap) { return max((min(max(len, 0), cap) + 31) >> 5, 1); }

// before, lens: of sequences lane * K .. lane * K + K - 1, without and with the token that the call appends.
// Every unit has `free` tiles that cost nothing in front of its real ones: a block that goes on to another unit has its merge and
// prologue to pay, and gets that many tiles less.  Units of equal tile counts are cut into as many even parts as there are blocks for,
// or kept whole, where that makes the busiest block's part shorter, merges included: above all where the sequences are short and the
// page table is wide, which the host's choice of this kernel goes by.  us a call in a graph, the other kernel / the cut that takes no
// notice of units / this (PoT-M4; costs of 0 to 64 tiles a merge were tried):
//   d = 64, 32 / 4 heads: 8 x 2048 of 32 768 tokens 9.3 / 11.1 / 9.8, 16 x 1024 of 16 384 10.1 / 11.5 / 8.2, 32 x 512 of 8192 12.1 / 11.6 / 8.0,
//     full 41.1 / 35.2 / 32.9;
//   d = 128, 32 / 8 heads: 24 x 256 of 4096 20.4 / 14.7 / 11.3, 32 x 512 of 8192 12.9 / 20.7 / 15.7, 32 x 2048 of 8192 32.9 / 37.6 / 34.0.
// (256 short units are what fills the other kernel's slots once, two units side by side on an SM and no splits; here a block has
// two of them one after the other.)
template <int D>
SA_D Stretch cut_stretch(const DecodeArgs& a, const int (&before)[kLaneSeqs], const int (&lens)[kLaneSeqs], int K, int lane, int blk) {
    const int B = a.batch, cap = a.max_pages * kPageTokens, R = a.Hkv * (a.G / a.gt), P = gridDim.x;
    int t[kLaneSeqs], sum = 0;
    bool same = true;
#pragma unroll
    for (int k = 0; k < kLaneSeqs; ++k) t[k] = k < K && lane * K + k < B ? stretch_tiles(lens[k], cap) : 0;
    const int T = __shfl_sync(0xffffffffu, t[0], 0);
#pragma unroll
    for (int k = 0; k < kLaneSeqs; ++k) same = same && (t[k] == 0 || t[k] == T);
    same = __all_sync(0xffffffffu, same);
    Stretch s;
    const int parts = same ? stream_parts(T, R * B, P, D) : 0;
    s.free = parts ? (parts - T % parts) % parts : stream_unit_cost(D);            // (even parts)
#pragma unroll
    for (int k = 0; k < kLaneSeqs; ++k) sum += t[k] ? t[k] + s.free : 0;
    int upto = sum;                                           // inclusive prefix over the lanes
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, upto, o);
        if (lane >= o) upto += x;
    }
    const int row = __shfl_sync(0xffffffffu, upto, 31), all = row * R;
    s.grain = parts ? (T + s.free) / parts : 1;
    const int grains = parts ? R * B * parts : all;
    s.each = grains / P * s.grain;
    s.more = grains % P;
    s.t0 = blk * s.each + min(blk, s.more) * s.grain;
    s.t1 = s.t0 + s.each + (blk < s.more ? s.grain : 0);
    s.y = min(s.t0 / row, R - 1);
    const int o = s.t0 - s.y * row;
    // the last sequence that begins at o or before
    int pre = upto - sum, found = 0, at = 0, tiles = 0, len = 0;
#pragma unroll
    for (int k = 0; k < kLaneSeqs; ++k)
        if (t[k] && pre <= o) {
            ++found;
            at = pre;
            tiles = t[k];
            len = before[k];
            pre += t[k] + s.free;
        }
    s.b = (int)__reduce_add_sync(0xffffffffu, (unsigned)found) - 1;
    const int owner = s.b / K;                                // (its last `found` is sequence b)
    s.start = s.y * row + __shfl_sync(0xffffffffu, at, owner);
    s.tiles = __shfl_sync(0xffffffffu, tiles, owner);
    s.len = __shfl_sync(0xffffffffu, len, owner);
    return s;
}
// The block whose stretch holds virtual tile t.
SA_D int block_of_tile(const Stretch& s, int t) {
    const int edge = s.more * (s.each + s.grain);
    return t < edge ? t / (s.each + s.grain) : s.more + (t - edge) / s.each;
}

// A unit that a block has been through: its rows are to be added.
struct UnitSums {
    bool any;
    int b, h0, u, first, blocks;  // sequence, first query head, place among the units; its first block, blocks that work on it
    bool marked;                  // a copy has not come
};

// What finish_units needs of the kernel's arguments and of the block's shared memory.
struct FinishArgs {
    float* O;
    float* partials;
    unsigned long long* counters;
    int32_t* plan;
    int GT, Hq, whole;
    float2* heads;                // [2][NW][8] {R, l}
    float* factors;               // [2][NW][8]
};
// Adds the rows of up to two units (the first one's {R, l} in the first half of heads), behind a block barrier: outputs of a
// unit that no other block has worked on, partials otherwise; the last block to leave a partial of a unit merges them, in the
// order of the blocks.
template <int D, int FMT, int NW>
SA_D void finish_units(const FinishArgs& a, const UnitSums& j0, const float* rows0, const UnitSums& j1, const float* rows1) {
    constexpr int NT = 32 * NW, kStep = TileMma<D, FMT, true, false>::kRowStep;
    constexpr float kValueScale = 1.0f / (1 << kWeightShift), kSumScale = FMT == FMT_FP16 ? kValueScale : 1.0f;
    const int GT = a.GT;
    if (threadIdx.x < 2 * NW * 8) {                           // every warp's 2^(R - R of the block's largest), and l times that
        float2* h = a.heads + threadIdx.x / (NW * 8) * (NW * 8);
        const int i = threadIdx.x % (NW * 8);
        float Rb = h[i % 8].x;
#pragma unroll
        for (int w = 1; w < NW; ++w) Rb = fmaxf(Rb, h[w * 8 + i % 8].x);
        const float f = pow2i_neg(__float2int_rn(h[i].x - Rb));
        a.factors[threadIdx.x] = f * kValueScale;
        h[i].y *= f * kSumScale;
    }
    __syncthreads();
#pragma unroll 1
    for (int n = 0; n < 2; ++n) {
        const UnitSums j = n ? j1 : j0;
        if (!j.any) continue;
        const float* rows = n ? rows1 : rows0;
        const float2* h = a.heads + n * (NW * 8);
        const float* fac = a.factors + n * (NW * 8);
        const bool whole = j.blocks == 1 && a.whole;
        float* out = whole ? a.O + ((size_t)j.b * a.Hq + j.h0) * D : a.partials + (size_t)((int)blockIdx.x + j.u) * GT * (D + 2) + 2;
        const int step = whole ? D : D + 2;
        for (int idx = threadIdx.x; idx < GT * (D / 2); idx += NT) {               // two dims of one head
            const int g = idx / (D / 2), col = idx % (D / 2);
            float x = 0.0f, y = 0.0f;
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                const float2 v = *reinterpret_cast<const float2*>(rows + (w * GT + g) * kStep + 2 * col);
                const float f = fac[w * 8 + g];
                x += v.x * f;
                y += v.y * f;
            }
            if (whole) {                                                           // no key at all: zeros; a copy that has not come: NaN
                float l = 0.0f;
#pragma unroll
                for (int w = 0; w < NW; ++w) l += h[w * 8 + g].y;
                const float inv = j.marked ? __int_as_float(0x7fc00000) : l == 0.0f ? 0.0f : 1.0f / l;
                x *= inv;
                y *= inv;
            }
            *reinterpret_cast<float2*>(out + g * step + 2 * col) = make_float2(x, y);
        }
        const int g = (int)threadIdx.x - (NT - 8);            // R and l (by the last warp: it has no more dims than the others)
        if (!whole && g >= 0 && g < GT) {
            float Rb = (float)kMNone, l = 0.0f;
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                Rb = fmaxf(Rb, h[w * 8 + g].x);
                l += h[w * 8 + g].y;
            }
            *reinterpret_cast<float2*>(out + g * step - 2) = j.marked ? make_float2(__int_as_float(0), __int_as_float(0x7fc00000))
                                                                      : make_float2(__int_as_float(__float2int_rn(Rb)), l);
        }
        if (!a.whole && threadIdx.x == 0 && j.first == (int)blockIdx.x) {          // for the merge kernel
            a.plan[2 * j.u] = j.first + j.u;
            a.plan[2 * j.u + 1] = j.blocks;
        }
    }
    const bool meet0 = a.whole && j0.any && j0.blocks > 1, meet1 = a.whole && j1.any && j1.blocks > 1;
    if (!meet0 && !meet1) return;
    __syncthreads();                                          // the block's partials are written
    int last = 0;
    if ((threadIdx.x == 0 && meet0) || (threadIdx.x == 32 && meet1)) {
        const UnitSums& j = threadIdx.x ? j1 : j0;
        __threadfence();
        const GlobalWord word{a.counters + j.u};
        last = last_to_arrive(word, j.blocks) ? 1 : 0;
        __threadfence();
        if (last) leave_at_rest(word, j.blocks);      // (behind the fence, which would wait for it)
    }
    const int merge0 = meet0 ? __syncthreads_or(threadIdx.x < 32 ? last : 0) : 0, merge1 = meet1 ? __syncthreads_or(threadIdx.x < 32 ? 0 : last) : 0;
#pragma unroll 1
    for (int n = 0; n < 2; ++n) {
        if (!(n ? merge1 : merge0)) continue;
        const UnitSums j = n ? j1 : j0;
        constexpr int kMost = 8;                              // partials whose loads are in flight together
        const int step = GT * (D + 2);
        for (int idx = threadIdx.x; idx < GT * (D / 2); idx += NT) {
            const int g = idx / (D / 2), col = idx % (D / 2);
            const float* row = a.partials + (size_t)(j.first + j.u) * step + g * (D + 2);
            int R = kMNone;
            float l = 0.0f, x = 0.0f, y = 0.0f;
            for (int k0 = 0; k0 < j.blocks; k0 += kMost) {
                float2 hd[kMost], v[kMost];
                int Rn = R;
#pragma unroll
                for (int k = 0; k < kMost; ++k) {
                    hd[k] = make_float2(__int_as_float(kMNone), 0.0f);
                    v[k] = make_float2(0.0f, 0.0f);
                    if (k0 + k < j.blocks) {
                        hd[k] = __ldcg(reinterpret_cast<const float2*>(row + (size_t)(k0 + k) * step));
                        v[k] = __ldcg(reinterpret_cast<const float2*>(row + (size_t)(k0 + k) * step + 2 + 2 * col));
                    }
                }
#pragma unroll
                for (int k = 0; k < kMost; ++k) Rn = max(Rn, __float_as_int(hd[k].x));
                const float fo = pow2i_neg(R - Rn);
                R = Rn;
                l *= fo;
                x *= fo;
                y *= fo;
#pragma unroll
                for (int k = 0; k < kMost; ++k) {
                    const float f = pow2i_neg(__float_as_int(hd[k].x) - Rn);       // (a partial without a key carries zeros)
                    l += hd[k].y * f;
                    x += v[k].x * f;
                    y += v[k].y * f;
                }
            }
            const float inv = l == 0.0f ? 0.0f : 1.0f / l;    // no key at all: zeros; a mark stays visible as NaN
            *reinterpret_cast<float2*>(a.O + ((size_t)j.b * a.Hq + j.h0 + g) * D + 2 * col) = make_float2(x * inv, y * inv);
        }
    }
}

// CODE, LOST: as in decode_mma_kernel.  FINE: as in TileMma.
template <int D, int FMT, int CODE, int NW, int NS, bool FINE, bool LOST>
__global__ void __maxnreg__(NW > 12 ? 128 : 168) decode_stream_kernel(const __grid_constant__ DecodeArgs a) {
    using SM = StreamSmem<D, FMT, NW, NS>;
    using Stage = typename SM::Stage;
    constexpr uint32_t kPolls = LOST ? (1u << 10) : kWaitLimit;
    extern __shared__ __align__(1024) uint8_t smem[];

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int GT = a.gt, chunks = a.G / GT, K = (a.batch + 31) >> 5;
    const uint32_t mbar0 = smem_addr(smem + SM::kMbarOff) + warp * NS * 8;
    const uint32_t stage0 = smem_addr(smem) + warp * NS * Stage::kBytes;
    int* len_s = reinterpret_cast<int*>(smem + SM::kLenOff);
    if (a.wait_first) pdl_wait();
    // Lengths without and with the token that the call appends, which needs a mapped page: a step cuts the tiles exactly as the
    // decode call on the extended cache does.
    int before[kLaneSeqs], lens[kLaneSeqs];
    auto read_length = [&](int k) { return k < K && lane * K + k < a.batch ? __ldcg(a.seq_lens + lane * K + k) : 0; };
    auto appends = [&](int k, int len) {
        if (!a.Knew || k >= K || lane * K + k >= a.batch || len < 0 || len / kPageTokens >= a.max_pages) return 0;
        return (unsigned)__ldcg(a.page_table + (size_t)(lane * K + k) * a.max_pages + len / kPageTokens) < (unsigned)a.n_pages ? 1 : 0;
    };
#pragma unroll
    for (int k = 0; k < kLaneSeqs; ++k) before[k] = read_length(k);
#pragma unroll
    for (int k = 0; k < kLaneSeqs; ++k) lens[k] = before[k] + appends(k, before[k]);
    if (lane == 0) {
#pragma unroll
        for (int s = 0; s < NS; ++s) mbar_init(mbar0 + s * 8, 1u);
        fence_mbar_init();
        fence_proxy_async();
    }
    __syncwarp();
    pdl_launch_dependents();

    TileMma<D, FMT, true, FINE> t;
    auto load_queries = [&](int y, int b) {
        const int h0 = (y / chunks) * a.G + (y % chunks) * GT, r = lane >> 2;
        t.load_queries(r < GT ? a.Q + ((size_t)b * a.Hq + h0 + r) * D : nullptr, lane, a.hadamard != 0, a.zscale);
    };
    Stretch s;
    int pidx_g[NS], pnew_g;
    bool again = LOST;                                        // (the test hook makes its first cut for another block)
#pragma unroll 1
    for (;;) {
        s = cut_stretch<D>(a, before, lens, K, lane, LOST && again ? (blockIdx.x + 1) % gridDim.x : blockIdx.x);
        // this warp's first tile: L2 is asked for it while the preceding kernel drains, its page is read behind the wait
        const int32_t* table = a.page_table + (size_t)s.b * a.max_pages;
        const int first_g = max(s.t0 - s.start - s.free, 0) + warp, end_g = min(min(s.t1 - s.start - s.free, s.tiles), a.max_pages * 2);
        const int p = first_g < end_g ? __ldcg(table + (first_g >> 1)) : -1;
        load_queries(s.y, s.b);                               // reads only Q, which no kernel of a decode step writes
        if (lane == 0 && (unsigned)p < (unsigned)a.n_pages)
            Stage::prefetch(a.pages + ((size_t)p * a.Hkv + s.y / chunks) * a.page_bytes, (first_g & 1) * 32, true);
        pdl_wait();                 // everything below reads what the preceding kernels in the stream wrote
        // one round trip where the cut stands
        int now[kLaneSeqs], grown[kLaneSeqs];
#pragma unroll
        for (int k = 0; k < kLaneSeqs; ++k) {
            now[k] = read_length(k);
            grown[k] = before[k] + appends(k, before[k]);
        }
#pragma unroll
        for (int i = 0; i < NS; ++i) pidx_g[i] = first_g + NW * i < end_g ? table[(first_g + NW * i) >> 1] : -1;
        const int lp_g = a.Knew && s.len >= 0 ? s.len / kPageTokens : a.max_pages;           // the new token's page
        pnew_g = lp_g < a.max_pages ? table[lp_g] : -1;
        if (a.Knew && lp_g < a.max_pages) {                   // its rows, for the warp that is to write it
            const int i = (s.len >> 5) - first_g;
            if (i >= 0 && (s.len >> 5) < end_g && i % NW == 0) {
                const size_t row = ((size_t)s.b * a.Hkv + s.y / chunks) * D;
                asm volatile("prefetch.global.L1 [%0];" ::"l"(a.Knew + row + lane * (D / 32)));
                asm volatile("prefetch.global.L1 [%0];" ::"l"(a.Vnew + row + lane * (D / 32)));
            }
        }
        bool stands = !again;
#pragma unroll
        for (int k = 0; k < kLaneSeqs; ++k) stands = stands && now[k] == before[k] && grown[k] == lens[k];
        if (__all_sync(0xffffffffu, stands)) break;
        again = false;
#pragma unroll
        for (int k = 0; k < kLaneSeqs; ++k) {
            before[k] = now[k];
            lens[k] = now[k] + appends(k, now[k]);
        }
    }
    // For the units to come: every warp writes the same lengths, and reads them back itself.
#pragma unroll
    for (int k = 0; k < kLaneSeqs; ++k)
        if (k < K && lane * K + k < a.batch) len_s[lane * K + k] = before[k];
    __syncwarp();

    float* rows_apart = reinterpret_cast<float*>(smem + SM::kRowOff);
    float* rows_alias = reinterpret_cast<float*>(smem);
    const bool apart = SM::apart(GT);
    float2* heads = reinterpret_cast<float2*>(smem + SM::kHeadOff);          // [2][NW][8] {R, l}
    float* factors = reinterpret_cast<float*>(smem + SM::kFactorOff);        // [2][NW][8]
    UnitSums held{};                                          // the unit whose rows wait in the place of their own
    int done = 0, turn = 0;                                   // tiles that this warp has taken (its stage buffer and phase); whose turn it is
    bool lost = false;                                        // a copy of this warp's has not come: its rows are marked from there on
    UnitSums unit{};
#pragma unroll 1
    for (bool next = false;; next = true) {
        const int kvh = s.y / chunks, h0 = kvh * a.G + (s.y % chunks) * GT, b = s.b;
        const int32_t* table = a.page_table + (size_t)b * a.max_pages;
        int len = s.len, tile_new = -1, pidx_new = -1;
        if (a.Knew) {
            const int lp = len / kPageTokens;
            pidx_new = !next ? pnew_g : (len >= 0 && lp < a.max_pages) ? table[lp] : -1;
            if (pidx_new >= 0 && pidx_new < a.n_pages) {
                tile_new = len >> 5;
                len += 1;
            }
        }
        if (next) s.tiles = stretch_tiles(len, a.max_pages * kPageTokens);
        const int lo = max(s.t0 - s.start - s.free, 0), hi = min(s.t1 - s.start - s.free, s.tiles);   // this block's tiles of the unit
        const bool more = s.t1 > s.start + s.free + s.tiles + s.free;        // a unit with tiles for this block follows
        unit.any = lo < hi;
        if (unit.any) {
            // ---- this warp's tiles (as in decode_mma_kernel), in turn through the units ----
            const int first = lo + (warp + NW - turn) % NW;
            turn = (turn + hi - lo) % NW;
            const int tile1 = min(hi, (min(len, a.max_pages * kPageTokens) + 31) >> 5);
            const int n_my = first < tile1 && !lost ? (tile1 - first + NW - 1) / NW : 0;
            const int i_new = (tile_new >= first && tile_new < tile1 && (tile_new - first) % NW == 0) ? (tile_new - first) / NW : -1;
            const uint8_t* pool = a.pages + (size_t)kvh * a.page_bytes + (first & 1) * Stage::kBytes;
            const uint32_t page_step = (uint32_t)a.Hkv * (uint32_t)a.page_bytes;
            auto issue = [&](int tile, int pidx, uint32_t st, uint32_t mb) {
                const bool mapped = (unsigned)pidx < (unsigned)a.n_pages;
                if (lane == 0 && !(LOST && tile == a.lost_tile && b == a.lost_b && kvh == a.lost_kvh)) {
                    if (mapped) Stage::issue(st, pool + (uint64_t)(uint32_t)pidx * page_step, 0, mb);
                    else mbar_arrive(mb);
                }
                return mapped ? len - tile * 32 : 0;
            };
            int n_keys[NS];
            if (next && lane == 0) fence_proxy_async();       // (the stages were read, as before every copy in the loop)
#pragma unroll
            for (int i = 0; i < NS; ++i)
                if (i < n_my && i != i_new) {
                    const int pidx = !next ? pidx_g[i] : table[(first + NW * i) >> 1];
                    n_keys[i] = issue(first + NW * i, pidx, stage0 + (done + i) % NS * Stage::kBytes, mbar0 + (done + i) % NS * 8);
                }
            if (i_new >= 0) {                                 // encode / quantise the token, write it into its page, copy its tile
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
                    if (i == i_new && i < n_my) n_keys[i] = issue(tile_new, pidx_new, stage0 + (done + i) % NS * Stage::kBytes, mbar0 + (done + i) % NS * 8);
            }
            if (next) load_queries(s.y, b);
            t.start();
            uint32_t st = stage0 + done % NS * Stage::kBytes, mb = mbar0 + done % NS * 8;
            const int32_t* next_page = table + ((first + NW * NS) >> 1);
            int tile = first;
            for (int i = 0; i < n_my; ++i, tile += NW, next_page += NW / 2) {
                // the page of the tile that will take this stage over, fetched while this one is worked on
                const int pidx_next = (i + NS < n_my) ? *next_page : -1;
                const uint32_t parity = (uint32_t)((done + i) / NS) & 1u;
                if (!__all_sync(0xffffffffu, mbar_try_wait(mb, parity)) && !__all_sync(0xffffffffu, mbar_wait_bounded(mb, parity, kPolls))) {
                    lost = true;
                    for (int k = 1; k < NS && i + k < n_my; ++k)
                        (void)mbar_wait_bounded(mbar0 + ((done + i + k) % NS) * 8, (uint32_t)((done + i + k) / NS) & 1u, kPolls);
                    break;
                }
                t.tile(a, st, n_keys[0], lane, b, h0, tile);
                __syncwarp();                                 // every lane is done with this stage
#pragma unroll
                for (int k = 0; k + 1 < NS; ++k) n_keys[k] = n_keys[k + 1];
                if (i + NS < n_my) {
                    if (lane == 0) fence_proxy_async();
                    n_keys[NS - 1] = issue(tile + NW * NS, pidx_next, st, mb);
                }
                if constexpr (NS == 2) {
                    st = 2 * stage0 + Stage::kBytes - st;
                    mb = 2 * mbar0 + 8 - mb;
                }
            }
            done += n_my;
            unit.b = b;
            unit.h0 = h0;
            unit.u = s.y * a.batch + b;
            unit.first = block_of_tile(s, s.start + s.free);
            unit.blocks = block_of_tile(s, s.start + s.free + s.tiles - 1) - unit.first + 1;
            unit.marked = lost;                               // (of this warp, so far)
            if (more && apart && !held.any) {                 // on to the next unit: the rows wait in the place of their own
                t.store_rows(heads, rows_apart, GT, lane, warp);
                held = unit;
            }
        }
        if (!more || (unit.any && !(held.any && held.u == unit.u))) {
            // ---- the last unit, or there is no other place for the rows: add them up, those that wait as well ----
            const bool alone = !held.any && apart && !more;   // the last unit's rows have a place of their own as well
            if (unit.any) {
                if (!alone) __syncthreads();                  // every warp is done with its stage buffers
                t.store_rows(heads + (alone ? 0 : NW * 8), alone ? rows_apart : rows_alias, GT, lane, warp);
            }
            unit.marked = __syncthreads_or(unit.any && unit.marked ? 1 : 0) != 0;
            if (held.any) held.marked = __syncthreads_or(held.marked ? 1 : 0) != 0;
            if (!more && a.arrivals && warp == NW - 1) bump_lengths(a, lane);      // every warp of the block has read the lengths
            UnitSums first_job = held, second_job = unit;
            if (alone) {
                first_job = unit;
                second_job.any = false;
            }
            finish_units<D, FMT, NW>(FinishArgs{a.O, a.partials, a.counters, a.plan, GT, a.Hq, a.whole, heads, factors}, first_job, rows_apart,
                                     second_job, rows_alias);
            if (!more) break;
            held.any = false;
            fence_proxy_async();                              // (the next copies land where the rows of all warps were)
            __syncthreads();
        }
        s.start += s.free + s.tiles;
        if (++s.b == a.batch) {
            s.b = 0;
            ++s.y;
        }
        s.len = len_s[s.b];
    }
}

template <int D, int FMT, int CODE, bool FINE, bool LOST>
static void launch_stream_as(const DecodeArgs& a, cudaStream_t s) {
    constexpr KernelShape sh = stream_shape(D, FMT == FMT_FP16);
    using SM = StreamSmem<D, FMT, sh.warps, sh.stages>;
    constexpr int most = SM::apart(8) ? SM::bytes(8) : SM::apart(4) ? SM::bytes(4) : SM::bytes(1);
    static_assert(most >= SM::bytes(1) && most >= SM::bytes(2) && most >= SM::bytes(4) && most >= SM::bytes(8), "for any number of heads");
    static OncePerDevice once;
    auto kernel = decode_stream_kernel<D, FMT, CODE, sh.warps, sh.stages, FINE, LOST>;
    if (!allow_shared(kernel, most, once)) return;            // (the caller asks for the last error)
    (void)launch_pdl(kernel, dim3((unsigned)a.stream), dim3(32 * sh.warps), (size_t)SM::bytes(a.gt), s, a);
}
template <int D, int FMT, int CODE, bool LOST = false>
static void launch_stream(const DecodeArgs& a, cudaStream_t s) {
    if (FMT != FMT_FP16 && !LOST && a.fine) launch_stream_as<D, FMT, CODE, FMT != FMT_FP16 && !LOST, LOST>(a, s);
    else launch_stream_as<D, FMT, CODE, false, LOST>(a, s);
}

}  // namespace sa
