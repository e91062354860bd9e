// Attention of one query group over one staged 32-key tile: what the decode kernels (sa_decode_mma.cuh,
// sa_decode_stream.cuh) do per tile, and the state a warp keeps over its tiles.
//
//   scores   exact integer products of the decoded key codes and the queries (sa_score_mma.cuh): keys x queries;
//   softmax  lane (r, c): keys r, r + 8, r + 16, r + 24 of queries 2 c, 2 c + 1.  The weight of a value row is
//            w = 2^(z - g - R) with an integer reference R per query that bounds z - g from above to within two bits
//            (z: logit in the log2 domain, 2^-g: the value's scale); the normaliser sums 2^(z - R).  R moves (and the
//            state is rescaled by the exact power of two) only when a weight would leave the range of binary16;
//   A.V      O^T[dims][queries] += V^T[dims][keys] w[keys][queries] as m16n8k16 products: INT8 values are exact in
//            binary16, every weight enters as the sum of two binary16 terms (22 significant bits for weights within
//            2^-17 of the largest, an absolute 2^-38 of it below), accumulation in FP32.  The weights reach the operand layout
//            through movmatrix, without shared memory.  (Binary16 values: one term, the weights rounded to binary16.)
#pragma once
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
template <int D, int FMT>
using MmaStage = TileStage<ScoreMma<D, FMT>::CH, FMT != FMT_FP16, FMT == FMT_FP16 ? 2 * D : D,
                           FMT == FMT_PLANAR1 ? 1 : FMT == FMT_PLANAR2 ? 2 : 0, D / 8>;

// LONG: for warps with many tiles.  Everything rare (a first tile, a reference that moves, slots past the sequence's end) is
// then out of the way of the other tiles, behind one vote, which is worth 2.5 % of a call with 55 tiles a warp; of calls with two,
// where every first tile takes the detour, it cost 2 to 5 %.
// FINE: the products of a tile are summed from zero and then added to the sums of the tiles before, rounded to nearest.  The
// matrix unit cuts its sums off, an error that grows with the number of products in one accumulator: 32 x 32 768 PoT-M4
// tokens, 55 tiles a warp, outputs 2.0e-6 too small (3.4e-6 with values of mean 1), with FINE 7e-8.  The
// additions cost 2 % at head_dim 64 (that call 98.3 -> 100.3 us, in a graph) and 1.5 - 7 % at 128, most where stretches are short
// (8 x 32 768 tokens, PoT-M4 88.8 -> 89.9, PoT-M1 planar 86.7 -> 89.5; 20 x 4096 36.6 -> 39.2), so warps with few tiles do without (see
// stream_is_fine).  (Sums put aside in tensor memory every 4 or 8 tiles instead: 1.2e-6 and 6 % at 4 tiles, a larger error at 8.)
template <int D, int FMT, bool LONG, bool FINE>
struct TileMma {
    using SC = ScoreMma<D, FMT>;
    using Stage = MmaStage<D, FMT>;
    static constexpr int MT = D / 16;              // 16-dim row tiles of O^T
    static constexpr bool kFp16 = FMT == FMT_FP16;
    static_assert(!(FINE && kFp16), "binary16 values: the weights' rounding is an error 100 times as large");
    static constexpr int kNever = 0x7fffffff;

    SC q;
    f32x2 qs;                                      // logit scale (Delta * log2(e) / sqrt(d) * unit of the scores) of queries 2 c, 2 c + 1
    f32x2 nR;                                      // - references of these queries (integers)
    f32x2 l;                                       // this lane's share of the normalisers
    float acc[MT][4];                              // O^T tiles: dims 16 mt + 2 r (c0, c1), + 1 (c2, c3) of queries 2 c, 2 c + 1
    bool seen;                                     // false: no key yet, the references are not set
    // LONG: tiles of fewer than `plain` keys are rare ones: all until the references are set, then those with slots past the
    // sequence's end.
    int plain;

    // Queries of the block: lane (r, c) reads row r (null: a zero query).
    SA_D void load_queries(const uint16_t* row, int lane, bool hadamard, float zscale) {
        const int c = lane & 3;
        const float d = q.load(row, lane, hadamard) * zscale;
        const float s0 = __shfl_sync(0xffffffffu, d, 8 * c), s1 = __shfl_sync(0xffffffffu, d, 8 * c + 4);
        qs = pack_f32x2(s0, s1);
    }
    SA_D void start() {
        nR = l = pack_f32x2(0.0f, 0.0f);
        seen = false;
        plain = kNever;
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[mt][e] = 0.0f;
    }

    // st: shared address of the staged tile, of whose keys the first n_valid count.  h0: the block's first query head.
    SA_D void tile(const DecodeArgs& a, uint32_t st, int n_valid, int lane, int b, int h0, int tile) {
        const int r = lane >> 2, c = lane & 3;
        float z[4][2], zh[SC::NACC == 2 ? 4 : 1][2];
        q.tile(st, st + Stage::kPlaneOff, lane, a.one, z, zh);
        if (a.dbg_scores) {                                   // parity tests only
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int e = 0; e < 2; ++e)
                    if (8 * j + r < n_valid && 2 * c + e < a.gt) {
                        int A = (int)(z[j][e] * a.score_unit);
                        if constexpr (SC::NACC == 2) A += (int)(zh[j][e] * a.score_unit);
                        a.dbg_scores[((size_t)b * a.Hq + h0 + 2 * c + e) * a.dbg_stride + (size_t)tile * 32 + 8 * j + r] =
                            (int)((uint32_t)A << a.f_extra);
                    }
        }
        // ---- logits and weights ----
        // The lane's two queries as packed FP32: the same arithmetic in half the instructions, and in few enough registers that
        // blocks of the merge kernel fit beside a full set of decode blocks: they are then there before the last of these ends.
        // A step of one sequence of 32 768 tokens took 10.85 us, 9.64 since.
        f32x2 zq[4];                                          // logit per score unit
        float vs[4];                                          // +- 2^(14 - g_j)
        uint32_t meta[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if constexpr (kFp16) {                            // no scales
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
            if constexpr (SC::NACC == 2) {                    // rounded once, like the conversion of one integer sum
                z[j][0] += zh[j][0];
                z[j][1] += zh[j][1];
            }
        }
        float p[4][2], w[4][2];
        __half2 h[4];
        auto weights = [&] {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float x0, x1;
                unpack_f32x2(ffma2(pack_f32x2(z[j][0], z[j][1]), zq[j], nR), &x0, &x1);
                p[j][0] = ex2_approx(x0);
                p[j][1] = ex2_approx(x1);
                w[j][0] = p[j][0] * fabsf(vs[j]);
                w[j][1] = p[j][1] * fabsf(vs[j]);
            }
        };
        // a weight beyond binary16 has become infinite: 0x7c00, the only value that 0x0400 carries into the sign bit
        auto round_weights = [&] {
#pragma unroll
            for (int j = 0; j < 4; ++j) h[j] = __floats2half2_rn(w[j][0], w[j][1]);
            const __half2 top = __hmax2(__hmax2(h[0], h[1]), __hmax2(h[2], h[3]));
            return ((*reinterpret_cast<const uint32_t*>(&top) + 0x04000400u) & 0x80008000u) != 0u;
        };
        bool rare = true;                                     // warp-uniform
        if constexpr (LONG) {
            rare = n_valid < plain;
            if (__builtin_expect(!rare, 1)) {
                weights();
                rare = __any_sync(0xffffffffu, round_weights());
            }
            rare = __builtin_expect(rare, 0);
        }
        if (rare) {
            bool move = !seen;                                // warp-uniform
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
                        float nR0, nR1;
                        unpack_f32x2(nR, &nR0, &nR1);
                        y0 = fmaxf(-nR0, y0);
                        y1 = fmaxf(-nR1, y1);
                        const float f0 = pow2i_neg(__float2int_rn(-nR0 - y0)), f1 = pow2i_neg(__float2int_rn(-nR1 - y1));
                        l = mul2(l, pack_f32x2(f0, f1));
#pragma unroll
                        for (int mt = 0; mt < MT; ++mt) {
                            acc[mt][0] *= f0;
                            acc[mt][1] *= f1;
                            acc[mt][2] *= f0;
                            acc[mt][3] *= f1;
                        }
                    }
                    nR = pack_f32x2(-y0, -y1);
                    seen = true;
                    plain = 32;
                }
                weights();
                if (n_valid < 32) {                           // the sequence's last tile: slots past its end may hold anything
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (8 * j + r >= n_valid) p[j][0] = p[j][1] = w[j][0] = w[j][1] = 0.0f;
                }
                move = __any_sync(0xffffffffu, round_weights());
                if (__builtin_expect(!move, 1)) break;
            }
        }
        uint32_t bh[4], bl[4];                                // operand fragments: keys 8 j + 2 c, + 1 of query r
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 hf = __half22float2(h[j]);
            bh[j] = movmatrix_trans(*reinterpret_cast<const uint32_t*>(&h[j]));
            if constexpr (kFp16) {
                // one term; the normaliser sums the same rounded weights, so the result is an exact weighted mean
                l = add2(l, pack_f32x2(hf.x, hf.y));
            } else {
                l = add2(l, pack_f32x2(p[j][0], p[j][1]));
                float x0, x1;                                 // what the first term leaves
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
            float own[4];                                     // FINE: the sums of this tile
            float(&sum)[4] = FINE ? own : acc[mt];
            if constexpr (kFp16) {                            // binary16 values: chunk 2 mt is rows r (dims 16 mt + r), chunk 2 mt + 1 rows r + 8
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
                if (FINE && k == 0) mma_f16_16816_first(sum, a0, a1, a2, a3, bh[0], bh[1]);
                else mma_f16_16816(sum, a0, a1, a2, a3, bh[2 * k], bh[2 * k + 1]);
                mma_f16_16816(sum, a0, a1, a2, a3, bl[2 * k], bl[2 * k + 1]);
            }
            if constexpr (FINE) {
                unpack_f32x2(add2(pack_f32x2(acc[mt][0], acc[mt][1]), pack_f32x2(own[0], own[1])), &acc[mt][0], &acc[mt][1]);
                unpack_f32x2(add2(pack_f32x2(acc[mt][2], acc[mt][3]), pack_f32x2(own[2], own[3])), &acc[mt][2], &acc[mt][3]);
            }
        }
    }

    // This warp's {R, l} of every query to heads ([warp][8]), its O to its rows ([warp][GT][kRowStep]), as they are (weights' scale
    // 2^14 included).  The row step keeps the lanes of a quad out of each other's banks.
    static constexpr int kRowStep = D + 8;
    SA_D void store_rows(float2* heads, float* rows, int GT, int lane, int warp) {
        const int r = lane >> 2, c = lane & 3;
        float l0, l1, nR0, nR1;
        unpack_f32x2(l, &l0, &l1);
        unpack_f32x2(nR, &nR0, &nR1);
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
            l0 += __shfl_xor_sync(0xffffffffu, l0, o);
            l1 += __shfl_xor_sync(0xffffffffu, l1, o);
        }
        if (r == 0) {
            heads[warp * 8 + 2 * c] = make_float2(seen ? -nR0 : (float)kMNone, l0);
            heads[warp * 8 + 2 * c + 1] = make_float2(seen ? -nR1 : (float)kMNone, l1);
        }
        float* row0 = rows + (warp * GT + 2 * c) * kRowStep;
#pragma unroll
        for (int e = 0; e < 2; ++e)
            if (2 * c + e < GT) {
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    float* row = row0 + e * kRowStep + 16 * mt;
                    if constexpr (kFp16) {
                        row[r] = acc[mt][e];
                        row[r + 8] = acc[mt][2 + e];
                    } else {
                        *reinterpret_cast<float2*>(row + 2 * r) = make_float2(acc[mt][e], acc[mt][2 + e]);
                    }
                }
            }
    }

    // The warps of a block, first half of their merge: R of every warp and query goes to ref_s ([warp][8]); behind a block
    // barrier every warp scales its state by the exact 2^(R - Rb), Rb the block's largest, and writes it to its row of red_s
    // ({unused, l, O[D]} of every warp and query).  Returns whether `failed` holds in any warp: then a bounded wait for a copy has
    // expired, and the caller marks the block's sum, from a register and not through the rows, which alias the stage buffers
    // (a copy that was merely late could still land in them).  after_barrier: what one warp does once all have come.
    template <int NW, typename After>
    SA_D bool merge_rows(float* ref_s, float (*red_s)[8][D + 2], int lane, int warp, bool failed, After after_barrier) {
        const int r = lane >> 2, c = lane & 3;
        float l0, l1, R0, R1;
        unpack_f32x2(l, &l0, &l1);
        unpack_f32x2(nR, &R0, &R1);
        R0 = -R0;
        R1 = -R1;
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
            l0 += __shfl_xor_sync(0xffffffffu, l0, o);
            l1 += __shfl_xor_sync(0xffffffffu, l1, o);
        }
        if (r == 0) {
            ref_s[warp * 8 + 2 * c] = seen ? R0 : (float)kMNone;
            ref_s[warp * 8 + 2 * c + 1] = seen ? R1 : (float)kMNone;
        }
        const bool poisoned = __syncthreads_or(failed ? 1 : 0) != 0;
        if (warp == 0) after_barrier();
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
        return poisoned;
    }
};

// The rows of merge_rows added in a fixed order, behind a block barrier: O[dim] of every head to sum_out (kSumStep floats a
// head), {R, l} of every head to head_out.
template <int D, int NW>
SA_D void sum_rows(const float* ref_s, float (*red_s)[8][D + 2], int GT, bool poisoned, float* sum_out, int sum_step, float* head_out, int head_step) {
    for (int idx = threadIdx.x; idx < GT * (D / 2); idx += 32 * NW) {              // two dims of one head
        const int g = idx / (D / 2), col = idx % (D / 2);
        float2 v = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const float2 x = *reinterpret_cast<const float2*>(&red_s[w][g][2 + 2 * col]);
            v.x += x.x;
            v.y += x.y;
        }
        *reinterpret_cast<float2*>(sum_out + g * sum_step + 2 * col) = v;
    }
    if (threadIdx.x >= 32 * NW - 8 && 8 - (32 * NW - (int)threadIdx.x) < GT) {     // R and l (by the last warp: it has no more dims than the others)
        const int g = 8 - (32 * NW - (int)threadIdx.x);
        float Rm = (float)kMNone, l = 0.0f;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            Rm = fmaxf(Rm, ref_s[w * 8 + g]);
            l += red_s[w][g][1];
        }
        *reinterpret_cast<float2*>(head_out + g * head_step) = poisoned ? make_float2(__int_as_float(0), __int_as_float(0x7fc00000))      // R = 0, l = NaN
                                                                        : make_float2(__int_as_float(__float2int_rn(Rm)), l);
    }
}

}  // namespace sa
