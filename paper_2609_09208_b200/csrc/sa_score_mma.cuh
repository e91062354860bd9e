// Integer scores of a 32-key tile as exact matrix products (the contraction of eq. (3) / (5) over head_dim).
//
// A tile's key codes are the A operand (rows = keys) and the block's up to 8 quantised queries the B operand of
// warp-level products; each code is decoded once, for all queries, into the small number it stands for:
//   byte / planar containers  (1 + j/2^k) * 2^(g - c) with its sign (g = 7 - e; 0 for the zero code).  Up to three
//                             mantissa bits (c = 7): as a binary16 value.  Sign, exponent field and mantissa field change
//                             places within the byte, four codes at a time, which makes it an FP8 (e4m3) value, and one
//                             conversion instruction turns two of those into binary16.  PoT-M4 (c = 127): as a bfloat16
//                             value, where the mantissa field has its place already.  Query integers (PoT-M4: times
//                             2^112) are values of the same type, so every product is exact in FP32, and so is the sum: it
//                             is a whole number of units 2^-(c - 1 + k) (PoT-M4: 2^-18) below 2^24
//                             (64 * 127 * 31 * 2^6 = 16 128 000 < 2^24 for PoT-M4).
//                             At head_dim 128 PoT-M4 could reach 2^25: its two halves are accumulated apart.
//   nibble container          2^(g - 1) <= 64 as an INT8 value: one byte permute looks four of them up, the sign bit of
//                             the nibble (the permute's replicate-sign mode over non-negative bytes) turning the
//                             others into 0; a second lookup with the signs flipped is multiplied by -q.  INT32 sums.
//   INT8 keys                 as stored.  INT32 sums.
//   binary16 keys             as stored, with the binary16 query; the sums are rounded like any FP32 sum.
// So the INT32 scores are those of the shift-and-add datapath (sa_datapath.cuh) bit for bit.  The decode is what a tile
// costs most: 7 instructions for four codes by way of FP8, 8 for PoT-M4 (11 as binary16).  The pipe of logic, shifts and
// permutes, which issues every other clock, is the fullest, the pipe of multiply-adds has room (62 and 20 % in a call of 32 x 32 768
// PoT-M4 tokens before; 63 and 19 now, with a fifth less time), so shifts to the left are multiplications by a constant that the
// compiler cannot see (`one`, the value 1, is a kernel argument).  With packed FP32 in the softmax (sa_tile_mma.cuh) that call of
// decode_mma_kernel, in a long run under the power cap, went from 128 to 123.3 us, 32 x 4096 tokens of head_dim 128 from 59.7 to 56.6.  Shifts to the right as the upper half of a product were slower (126.6), FP8 operands of
// the product itself, which are exact too, far slower (116 -> 147).
//
// Fragments: lane (r, c) = (lane / 4, lane % 4) holds the c-th 32-bit word of a 16-byte code chunk of keys r, r + 8,
// r + 16, r + 24 (one ldmatrix.x4 per chunk: 8 keys x 16 bytes are 128 contiguous bytes, no bank conflict).  The order of
// the elements along the contraction is free as long as the queries are packed in the same order.
#pragma once
#include <cuda_bf16.h>

#include "sa_common.cuh"
#include "sa_datapath.cuh"
#include "sa_mma.cuh"
#include "sa_quant.cuh"

namespace sa {

// FMT_FP16: the unquantised cache; FMT_BYTE3: the byte container of the codes with at most three mantissa bits (all but PoT-M4)
enum ScoreFormat { FMT_BYTE = 0, FMT_NIBBLE = 1, FMT_PLANAR1 = 2, FMT_PLANAR2 = 3, FMT_INT8 = 4, FMT_BYTE3 = 5, FMT_FP16 = 6 };

// Codes I, I + 1 of a word of the byte container (sign << 7 | mantissa << 3 | g) as a pair of bfloat16 values.  With the byte in
// both halves of its value, the mantissa field and the sign are where bfloat16 has them; g moves to bits 9..7.
template <int I>
SA_D uint32_t byte_codes_to_bf16(uint32_t w, uint32_t one) {
    const uint32_t h = __byte_perm(w, 0u, I ? 0x3322u : 0x1100u);
    return (h & 0x80788078u) | ((h * (one * 128u)) & 0x03800380u);
}
// Four codes of the byte container with at most three mantissa bits as FP8 values (sign << 7 | g << 3 | mantissa >> 1).
SA_HD uint32_t byte_codes_to_fp8(uint32_t w, uint32_t one) {
    return (w & 0x80808080u) | ((w * (one * 8u)) & 0x38383838u) | ((w >> 4) & 0x07070707u);
}
// FP8 values 0 and 1 (HIGH: 2 and 3) of a word as a pair of binary16 values.
template <bool HIGH>
SA_D uint32_t fp8_to_half2(uint32_t f) {
    uint32_t h;
    if constexpr (HIGH) asm("{.reg .b16 l, h; mov.b32 {l, h}, %1; cvt.rn.f16x2.e4m3x2 %0, h;}" : "=r"(h) : "r"(f));
    else asm("{.reg .b16 l, h; mov.b32 {l, h}, %1; cvt.rn.f16x2.e4m3x2 %0, l;}" : "=r"(h) : "r"(f));
    return h;
}
// Even (ODD: odd) elements of a word of nibbles (sign << 3 | g) as FP8 powers of two with their signs.
template <bool ODD>
SA_HD uint32_t nibble_codes_to_fp8(uint32_t w, uint32_t one) {
    return ODD ? ((w & 0x80808080u) | ((w >> 1) & 0x38383838u)) : (((w * (one * 16u)) & 0x80808080u) | ((w * (one * 8u)) & 0x38383838u));
}
// The mantissa bits of the even elements in a byte of a bit plane (odd ones: of the byte >> 1), bit 2 i to bit AT of byte
// i: the product places copies of the byte at offsets 6 apart, the mask keeps the wanted bit of each.
template <int AT>
SA_HD uint32_t plane_bits(uint32_t p) {
    return ((p & 0x55u) * (0x00041041u << AT)) & (0x01010101u << AT);
}
// INT8 values of two keys of one dimension (bytes 0 and 2, ODD: 1 and 3) as a pair of binary16 values: the biased byte
// v + 128 in the low mantissa bits of 1024, minus 1152 (exact).
template <bool ODD>
SA_D uint32_t int8_to_half2(uint32_t x) {
    const uint32_t y = ODD ? x >> 8 : x;
    uint32_t h = (y & 0x00ff00ffu) ^ 0x64806480u;
    asm("add.rn.f16x2 %0, %0, %1;" : "+r"(h) : "r"(0xe480e480u));
    return h;
}

// The quantised queries of a block as B fragments in registers of every warp: lane (r, c) prepares query r.
// E consecutive elements per lane and chunk: 2, 4 or 8 (chunks of 8, 16 or 32 elements).
template <int D, int FMT>
struct ScoreMma {
    static constexpr bool kInt = (FMT == FMT_NIBBLE || FMT == FMT_INT8);
    static constexpr bool kDense = (FMT == FMT_NIBBLE || FMT == FMT_PLANAR1 || FMT == FMT_PLANAR2);
    static constexpr int E = FMT == FMT_FP16 ? 2 : kDense ? 8 : 4;
    static constexpr int CH = D / (4 * E);                        // code chunks
    static constexpr int NACC = (FMT == FMT_BYTE && D == 128) ? 2 : 1;
    static constexpr int NB = kInt ? D / 16 : D / 8;              // registers of B fragments
    uint32_t q[NB];
    uint32_t qn[FMT == FMT_NIBBLE ? NB : 1];                      // -q

    // Quantises query r of this lane's fragment row (row: its D binary16 elements; null: a zero query).  Same
    // arithmetic, in the same order, as quantise_query_vec: rotation with strides 1, 2, ..., largest magnitude,
    // IEEE divide, round half to even.  Returns Delta.
    SA_D float load(const uint16_t* row, int lane, bool hadamard) {
        const int c = lane & 3;
        if constexpr (FMT == FMT_FP16) {                          // nothing to quantise
#pragma unroll
            for (int k = 0; k < CH; ++k) q[k] = row ? *reinterpret_cast<const uint32_t*>(row + k * 8 + c * 2) : 0u;
            return 1.0f;
        } else {
            return quantise(row, c, hadamard);
        }
    }
    SA_D float quantise(const uint16_t* row, int c, bool hadamard) {
        float x[CH][E];
#pragma unroll
        for (int k = 0; k < CH; ++k)
#pragma unroll
            for (int i = 0; i < E; i += 4) {
                uint2 w = make_uint2(0u, 0u);
                if (row) w = *reinterpret_cast<const uint2*>(row + k * 4 * E + c * E + i);
                x[k][i] = half_bits_to_float(w.x & 0xffffu);
                x[k][i + 1] = half_bits_to_float(w.x >> 16);
                x[k][i + 2] = half_bits_to_float(w.y & 0xffffu);
                x[k][i + 3] = half_bits_to_float(w.y >> 16);
            }
        if (hadamard) rotate(x, c);
        float amax = 0.0f;
#pragma unroll
        for (int k = 0; k < CH; ++k)
#pragma unroll
            for (int i = 0; i < E; ++i) amax = fmaxf(amax, fabsf(x[k][i]));
        amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 1));
        amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 2));
        const float inv = amax == 0.0f ? 0.0f : __fdiv_rn(127.0f, amax);
        int v[CH][E];
#pragma unroll
        for (int k = 0; k < CH; ++k)
#pragma unroll
            for (int i = 0; i < E; ++i) v[k][i] = max(-127, min(127, __float2int_rn(__fmul_rn(x[k][i], inv))));
        pack(v);
        return __fdiv_rn(amax, 127.0f);
    }

    // D-element Walsh-Hadamard transform of the quad's four lanes (element k * 4E + c * E + i), rounded to binary16.
    SA_D static void rotate(float (&x)[CH][E], int c) {
#pragma unroll
        for (int h = 1; h < E; h <<= 1)
#pragma unroll
            for (int k = 0; k < CH; ++k)
#pragma unroll
                for (int i = 0; i < E; ++i)
                    if ((i & h) == 0) {
                        const float a = x[k][i], b = x[k][i + h];
                        x[k][i] = __fadd_rn(a, b);
                        x[k][i + h] = __fsub_rn(a, b);
                    }
#pragma unroll
        for (int h = 1; h < 4; h <<= 1)
#pragma unroll
            for (int k = 0; k < CH; ++k)
#pragma unroll
                for (int i = 0; i < E; ++i) {
                    const float o = __shfl_xor_sync(0xffffffffu, x[k][i], h);
                    x[k][i] = (c & h) ? __fsub_rn(o, x[k][i]) : __fadd_rn(x[k][i], o);
                }
#pragma unroll
        for (int h = 1; h < CH; h <<= 1)
#pragma unroll
            for (int k = 0; k < CH; ++k)
                if ((k & h) == 0)
#pragma unroll
                    for (int i = 0; i < E; ++i) {
                        const float a = x[k][i], b = x[k + h][i];
                        x[k][i] = __fadd_rn(a, b);
                        x[k + h][i] = __fsub_rn(a, b);
                    }
        const float scale = (D == 64) ? 0.125f : 0.088388346f;    // 1/sqrt(64), 1/sqrt(128)
#pragma unroll
        for (int k = 0; k < CH; ++k)
#pragma unroll
            for (int i = 0; i < E; ++i) x[k][i] = __half2float(__float2half_rn(__fmul_rn(x[k][i], scale)));
    }

    SA_D static uint32_t b4(int a, int b, int c, int d) {
        return (uint32_t)(a & 0xff) | ((uint32_t)(b & 0xff) << 8) | ((uint32_t)(c & 0xff) << 16) | ((uint32_t)d << 24);
    }
    SA_D static uint32_t h2(int lo, int hi) {                     // |integers| <= 127: exact
        const __half2 h = __floats2half2_rn((float)lo, (float)hi);
        return *reinterpret_cast<const uint32_t*>(&h);
    }
    // |integers| <= 127 times 2^112: exact.  The keys' exponent field starts at 2^-127; the factor makes the unit 2^-18.
    SA_D static uint32_t bf2(int lo, int hi) {
        const __nv_bfloat162 h = __floats2bfloat162_rn((float)lo * 0x1p112f, (float)hi * 0x1p112f);
        return *reinterpret_cast<const uint32_t*>(&h);
    }
    // The order of the elements along the contraction: that of tile() below.
    SA_D void pack(const int (&v)[CH][E]) {
#pragma unroll
        for (int k = 0; k < CH; ++k) {
            if constexpr (FMT == FMT_BYTE) {
                q[2 * k] = bf2(v[k][0], v[k][1]);
                q[2 * k + 1] = bf2(v[k][2], v[k][3]);
            } else if constexpr (FMT == FMT_BYTE3) {
                q[2 * k] = h2(v[k][0], v[k][1]);
                q[2 * k + 1] = h2(v[k][2], v[k][3]);
            } else if constexpr (FMT == FMT_INT8) {
                q[k] = b4(v[k][0], v[k][1], v[k][2], v[k][3]);
            } else if constexpr (FMT == FMT_NIBBLE) {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    q[2 * k + i] = b4(v[k][4 * i], v[k][4 * i + 1], v[k][4 * i + 2], v[k][4 * i + 3]);
                    qn[2 * k + i] = b4(-v[k][4 * i], -v[k][4 * i + 1], -v[k][4 * i + 2], -v[k][4 * i + 3]);
                }
            } else {
#pragma unroll
                for (int i = 0; i < 2; ++i) {                     // even, then odd elements
                    q[4 * k + 2 * i] = h2(v[k][i], v[k][2 + i]);
                    q[4 * k + 2 * i + 1] = h2(v[k][4 + i], v[k][6 + i]);
                }
            }
        }
    }

    // Scores of the 32 keys of a staged tile: sc[j][e], j = 2 t + h: key 16 t + 8 h + r, query 2 c + e, in units of
    // 2^-(6 + k) (PoT-M4: 2^-18; integer formats: 1).  st: shared address of the tile's codes; planes: its mantissa bit planes.
    // hi[][]: the part of dimensions 64 .. 127 of NACC == 2 (not yet added).  one: DecodeArgs::one.
    SA_D void tile(uint32_t st, uint32_t planes, int lane, uint32_t one, float (&sc)[4][2], float (&hi)[NACC == 2 ? 4 : 1][2]) const {
        const uint32_t row = st + lane * 16;
        if constexpr (kInt) {
            int d[2][4] = {};
            if constexpr (FMT == FMT_INT8) {
#pragma unroll
                for (int k = 0; k < CH; k += 2) {
                    uint32_t a[4], b[4];
                    ldmatrix_x4(a, row + k * 512);
                    ldmatrix_x4(b, row + (k + 1) * 512);
#pragma unroll
                    for (int t = 0; t < 2; ++t) mma_s8_16832(d[t], a[2 * t], a[2 * t + 1], b[2 * t], b[2 * t + 1], q[k], q[k + 1]);
                }
            } else {
#pragma unroll
                for (int k = 0; k < CH; ++k) {
                    uint32_t w[4];
                    ldmatrix_x4(w, row + k * 512);
#pragma unroll
                    for (int t = 0; t < 2; ++t) {
                        const uint32_t w0 = w[2 * t], w1 = w[2 * t + 1], n0 = w0 ^ 0x88888888u, n1 = w1 ^ 0x88888888u;
                        mma_s8_16832(d[t], lookup(w0), lookup(w1), lookup(w0 >> 16), lookup(w1 >> 16), q[2 * k], q[2 * k + 1]);
                        mma_s8_16832(d[t], lookup(n0), lookup(n1), lookup(n0 >> 16), lookup(n1 >> 16), qn[2 * k], qn[2 * k + 1]);
                    }
                }
            }
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int e = 0; e < 4; ++e) sc[2 * t + (e >> 1)][e & 1] = (float)d[t][e];      // below 2^24: exact
        } else {
            float d[2 * NACC][4] = {};
            if constexpr (FMT == FMT_FP16) {
#pragma unroll
                for (int k = 0; k < CH; k += 2) {
                    uint32_t w0[4], w1[4];
                    ldmatrix_x4(w0, row + k * 512);
                    ldmatrix_x4(w1, row + (k + 1) * 512);
#pragma unroll
                    for (int t = 0; t < 2; ++t) mma_f16_16816(d[t], w0[2 * t], w0[2 * t + 1], w1[2 * t], w1[2 * t + 1], q[k], q[k + 1]);
                }
            } else if constexpr (!kDense) {
#pragma unroll
                for (int k = 0; k < CH; ++k) {
                    uint32_t w[4];
                    ldmatrix_x4(w, row + k * 512);
#pragma unroll
                    for (int t = 0; t < 2; ++t) {
                        float(&acc)[4] = d[(NACC == 2 && k >= CH / 2 ? 2 : 0) + t];
                        if constexpr (FMT == FMT_BYTE) {
                            mma_bf16_16816(acc, byte_codes_to_bf16<0>(w[2 * t], one), byte_codes_to_bf16<0>(w[2 * t + 1], one),
                                           byte_codes_to_bf16<2>(w[2 * t], one), byte_codes_to_bf16<2>(w[2 * t + 1], one), q[2 * k], q[2 * k + 1]);
                        } else {
                            const uint32_t f0 = byte_codes_to_fp8(w[2 * t], one), f1 = byte_codes_to_fp8(w[2 * t + 1], one);
                            mma_f16_16816(acc, fp8_to_half2<false>(f0), fp8_to_half2<false>(f1), fp8_to_half2<true>(f0), fp8_to_half2<true>(f1),
                                          q[2 * k], q[2 * k + 1]);
                        }
                    }
                }
            } else {
#pragma unroll
                for (int k = 0; k < CH; ++k) {
                    uint32_t w[4];
                    ldmatrix_x4(w, row + k * 512);
#pragma unroll
                    for (int t = 0; t < 2; ++t) {
                        uint32_t f[2][2];                                      // [key r / r + 8 of the half][even / odd elements]
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int j = 2 * t + h;
                            f[h][0] = nibble_codes_to_fp8<false>(w[j], one);
                            f[h][1] = nibble_codes_to_fp8<true>(w[j], one);
                            const uint32_t pa = planes + (8 * j + (lane >> 2)) * (D / 8) + 4 * k + (lane & 3);
                            uint32_t p = lds_u8(pa);
                            f[h][0] |= plane_bits<FMT == FMT_PLANAR1 ? 2 : 1>(p);
                            f[h][1] |= plane_bits<FMT == FMT_PLANAR1 ? 2 : 1>(p >> 1);
                            if constexpr (FMT == FMT_PLANAR2) {
                                p = lds_u8(pa + 32 * (D / 8));
                                f[h][0] |= plane_bits<2>(p);
                                f[h][1] |= plane_bits<2>(p >> 1);
                            }
                        }
#pragma unroll
                        for (int i = 0; i < 2; ++i)
                            mma_f16_16816(d[t], fp8_to_half2<false>(f[0][i]), fp8_to_half2<false>(f[1][i]), fp8_to_half2<true>(f[0][i]),
                                          fp8_to_half2<true>(f[1][i]), q[4 * k + 2 * i], q[4 * k + 2 * i + 1]);
                    }
                }
            }
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    sc[2 * t + (e >> 1)][e & 1] = d[t][e];
                    if constexpr (NACC == 2) hi[2 * t + (e >> 1)][e & 1] = d[2 + t][e];
                }
        }
    }

private:
    SA_D static uint32_t lookup(uint32_t w) {                     // 2^(g - 1) of four nibbles, 0 where the sign bit is set
        uint32_t d;
        asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(0x04020100u), "r"(0x40201008u), "r"(w));
        return d;
    }
};

}  // namespace sa
