// Cache-write side of the library: key encode, query and value quantisation, append, bulk
// fill and the unpack test hook.  One warp handles one head vector; lane l owns the
// head_dim / 32 consecutive elements starting at l * (head_dim / 32).
#include "sa_common.cuh"
#include "sa_cache_write.cuh"
#include "sa_quant.cuh"

namespace sa {

// -------------------------------------------------------------------------------------------
// sa_encode_keys: canonical bytes + scales.
// -------------------------------------------------------------------------------------------
template <int D, int K>
__global__ void __launch_bounds__(128) encode_keys_kernel(const uint16_t* __restrict__ Kin, int64_t n_vec,
                                                          uint8_t* __restrict__ codes,
                                                          uint16_t* __restrict__ scales, int hadamard) {
    constexpr int EPL = D / 32;
    const int lane = threadIdx.x & 31;
    const int64_t v = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
    if (v >= n_vec) return;
    uint32_t bits[EPL];
    load_vec_bits<EPL>(Kin + v * D, lane, bits);
    uint8_t c[EPL];
    uint32_t smax;
    if constexpr (K == 8) smax = encode_key_int8_vec<EPL>(bits, lane, hadamard != 0, c);
    else smax = encode_key_vec<EPL, K>(bits, lane, hadamard != 0, c);
    store_bytes<EPL>(codes + v * D + lane * EPL, c);
    if (lane == 0) scales[v] = (uint16_t)smax;
}

// -------------------------------------------------------------------------------------------
// sa_quantise_query
// -------------------------------------------------------------------------------------------
template <int D>
__global__ void __launch_bounds__(128) quantise_query_kernel(const uint16_t* __restrict__ Q, int64_t n_vec,
                                                             int8_t* __restrict__ qhat,
                                                             float* __restrict__ delta, int hadamard) {
    constexpr int EPL = D / 32;
    const int lane = threadIdx.x & 31;
    const int64_t v = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
    if (v >= n_vec) return;
    uint32_t bits[EPL];
    load_vec_bits<EPL>(Q + v * D, lane, bits);
    int q[EPL];
    const float dl = quantise_query_vec<EPL>(bits, lane, hadamard != 0, q);
    uint8_t c[EPL];
#pragma unroll
    for (int i = 0; i < EPL; ++i) c[i] = (uint8_t)(int8_t)q[i];
    store_bytes<EPL>(reinterpret_cast<uint8_t*>(qhat) + v * D + lane * EPL, c);
    if (lane == 0) delta[v] = dl;
}

// -------------------------------------------------------------------------------------------
// sa_quantise_values
// -------------------------------------------------------------------------------------------
template <int D>
__global__ void __launch_bounds__(128) quantise_values_kernel(const uint16_t* __restrict__ V, int64_t n_vec,
                                                              int8_t* __restrict__ vhat,
                                                              int8_t* __restrict__ g) {
    constexpr int EPL = D / 32;
    const int lane = threadIdx.x & 31;
    const int64_t v = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
    if (v >= n_vec) return;
    uint32_t bits[EPL];
    load_vec_bits<EPL>(V + v * D, lane, bits);
    uint8_t c[EPL];
    const int gg = quantise_value_vec<EPL>(bits, c);
    store_bytes<EPL>(reinterpret_cast<uint8_t*>(vhat) + v * D + lane * EPL, c);
    if (lane == 0) g[v] = (int8_t)gg;
}

// sa_append_kv: one block per sequence; warps loop over the KV heads.
template <int D, int MODE>
__global__ void __launch_bounds__(128) append_kernel(CacheArgs a, const uint16_t* __restrict__ Knew,
                                                     const uint16_t* __restrict__ Vnew, int bump) {
    pdl_wait();                 // earlier kernels in the stream may still be reading this cache
    pdl_launch_dependents();
    const int b = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int len = a.seq_lens[b];
    const bool ok = len >= 0 && page_block(a, b, len / kPageTokens, 0) != nullptr;
    if (ok) {
        for (int h = warp; h < a.Hkv; h += 4) {
            uint8_t* block = page_block(a, b, len / kPageTokens, h);
            const size_t row = ((size_t)b * a.Hkv + h) * D;
            write_token<D, MODE>(block, a, len % kPageTokens, lane, Knew + row, Vnew + row);
        }
    }
    __syncthreads();   // every warp has read seq_lens[b] before it changes
    if (ok && bump && threadIdx.x == 0) a.seq_lens[b] = len + 1;
}

// sa_fill_kv.  One warp takes the keys or the values of one KV head for the 32 tokens of half a page.  It loads whole 128-byte
// lines and turns them in shared memory, so that lane = token: a thread has its whole head vector (no shuffles for the largest
// magnitude or the rotation), and as the chunks of the 32 tokens follow one another in the page, the warp's stores are
// 512 contiguous bytes per chunk.  (Each thread loading its own row meant 32 lines per load instruction.)  All sequences of a
// call go in one launch.  Large calls are bound by the encoder on the ALU pipe (82 % before signs and value bytes were handled
// four at a time), binary16 by memory; the smallest by the fetch of code that every warp runs once, hence rolled loops where
// 64 unrolled elements are tens of kilobytes (PoT-4's short code is better off with 32 at a time).  Measured on PoT-M4 /
// PoT-4 / binary16, us: 32 tokens of 4 heads 4.7 / 3.5 / 2.0 -> 3.0 / 2.5 / 1.8, four prompts of 18 384 tokens 12.3 / 10.0 / 8.4
// -> 9.1 / 7.4 / 7.5, 8 x 32768 tokens 109 / 90 / 91 -> 102 / 89 / 81 (81 us are the copy rate).
constexpr int kFillBatch = 64;            // sequences per launch
struct FillSeqs {
    int64_t row0[kFillBatch];             // first row of the sequence in K / V
    int tiles[kFillBatch + 1];            // 32-token tiles ahead of it
    int len[kFillBatch];
    int b0, n;                            // sequences b0 .. b0 + n - 1
};

// Walsh-Hadamard rotation of a whole head vector in one thread, as hadamard_warp (the same butterflies in the same order).
template <int D>
SA_D void hadamard_thread(uint32_t (&h)[D / 2]) {
    float x[D];
#pragma unroll
    for (int i = 0; i < D / 2; ++i) {
        x[2 * i] = half_bits_to_float(h[i] & 0xffffu);
        x[2 * i + 1] = half_bits_to_float(h[i] >> 16);
    }
#pragma unroll
    for (int st = 1; st < D; st <<= 1)
#pragma unroll
        for (int i = 0; i < D; ++i)
            if ((i & st) == 0) {
                const float a = x[i], b = x[i + st];
                x[i] = __fadd_rn(a, b);
                x[i + st] = __fsub_rn(a, b);
            }
    const float scale = (D == 64) ? 0.125f : 0.088388346f;
#pragma unroll
    for (int i = 0; i < D / 2; ++i)
        h[i] = (uint32_t)__half_as_ushort(__float2half_rn(__fmul_rn(x[2 * i], scale))) |
               ((uint32_t)__half_as_ushort(__float2half_rn(__fmul_rn(x[2 * i + 1], scale))) << 16);
}

// The vector of one token -> its place in the half page `half` (t: token within it).
SA_D float2 half2_bits_to_float2(uint32_t x) { return __half22float2(*reinterpret_cast<const __half2*>(&x)); }

// One thread's vector in the warp's shared buffer (16-byte chunk i of row t at chunk i ^ (t & 7), so that neither the rows'
// owners nor the coalesced writes meet a bank conflict): its largest magnitude, then its elements 8 at a time.  KEEP: rotated,
// in registers.
template <int D, bool KEEP>
struct VecRow {
    const uint4* row;
    int x7;
    uint32_t h[KEEP ? D / 2 : 1];
    uint32_t top = 0;
    SA_D VecRow(const uint4* buffer, int t) : row(buffer + t * (D / 8)), x7(t & 7) {
        if constexpr (KEEP) {
#pragma unroll
            for (int i = 0; i < D / 8; ++i) {
                const uint4 v = row[i ^ x7];
                h[4 * i] = v.x, h[4 * i + 1] = v.y, h[4 * i + 2] = v.z, h[4 * i + 3] = v.w;
            }
            hadamard_thread<D>(h);
#pragma unroll
            for (int i = 0; i < D / 2; ++i) top = __vmaxu2(top, h[i] & 0x7fff7fffu);      // two magnitudes at a time; they order like their bits
        } else {
#pragma unroll
            for (int i = 0; i < D / 8; ++i) {
                const uint4 v = row[i ^ x7];
                top = __vmaxu2(__vmaxu2(top, __vmaxu2(v.x & 0x7fff7fffu, v.y & 0x7fff7fffu)), __vmaxu2(v.z & 0x7fff7fffu, v.w & 0x7fff7fffu));
            }
        }
    }
    SA_D uint32_t max_bits() const { return max(top & 0xffffu, top >> 16); }
    SA_D void get(int i, uint32_t* x) const {
        if constexpr (KEEP) {
#pragma unroll
            for (int e = 0; e < 4; ++e) x[e] = h[4 * i + e];
        } else {
            const uint4 v = row[i ^ x7];
            x[0] = v.x, x[1] = v.y, x[2] = v.z, x[3] = v.w;
        }
    }
};
template <int D, int MODE, bool HAD>
SA_D void fill_keys(uint8_t* half, const CacheArgs& a, int t, const uint4* src) {
    constexpr bool NIB = MODE >= 8 && MODE <= 10;
    constexpr int K = MODE == 32 ? 8 : NIB ? MODE - 8 : MODE;
    VecRow<D, HAD> row(src, t);
    const uint32_t smax = row.max_bits();
    const KeyScale ks = key_scale(smax);
    const float amax = half_bits_to_float(smax);
    const float inv8 = (K == 8 && amax != 0.0f) ? __fdiv_rn(127.0f, amax) : 0.0f;
    auto place = [&](float x) -> uint32_t {                   // 0 for the zero code
        const uint32_t p = encode_place(K, x, ks);
        return p < (1u << K) ? 0u : p;
    };
    uint8_t* dst = half + a.kcode_off + (size_t)t * 16;
    if constexpr (!NIB) {
#pragma unroll(HAD ? D / 16 : 1)
        for (int c = 0; c < D / 16; ++c) {
            uint32_t x[8], w[4];
            row.get(2 * c, x);
            row.get(2 * c + 1, x + 4);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 f[2] = {half2_bits_to_float2(x[2 * i]), half2_bits_to_float2(x[2 * i + 1])};
                const float e[4] = {f[0].x, f[0].y, f[1].x, f[1].y};
                w[i] = 0u;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if constexpr (K == 8) {
                        const int q = __float2int_rn(__fmul_rn(e[k], inv8));
                        w[i] |= ((uint32_t)max(-127, min(127, q)) & 0xffu) << (8 * k);
                    } else {
                        const uint32_t p = place(e[k]);       // -> mantissa field << 3 | g
                        w[i] |= (((p << (7 - K)) & (0x7fu & (0x7fu << (7 - K)))) | (p >> K)) << (8 * k);
                    }
                }
                // the four signs at once, kept beside nonzero bytes only
                if constexpr (K != 8) w[i] |= __byte_perm(x[2 * i], x[2 * i + 1], 0x7531) & 0x80808080u & (w[i] + 0x7f7f7f7fu);
            }
            *reinterpret_cast<uint4*>(dst + (size_t)(c * kTileTokens) * 16) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    } else {
        constexpr int P = K > 0 && K < 8 ? K : 1;
        uint32_t w[4] = {}, plane[P] = {};                    // the chunk and the mantissa bits of its 32 elements, filled from the top
#pragma unroll(HAD ? D / 8 : K == 0 ? 4 : 1)
        for (int i = 0; i < D / 8; ++i) {
            uint32_t x[4], next = 0u;
            row.get(i, x);
#pragma unroll
            for (int bit = 0; bit < P; ++bit) plane[bit] >>= 8;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float2 f = half2_bits_to_float2(x[e >> 1]);
                const uint32_t p = place((e & 1) ? f.y : f.x);
                next |= (p >> K) << (4 * e);
                if constexpr (K > 0)
#pragma unroll
                    for (int bit = 0; bit < K; ++bit) plane[bit] |= ((p >> bit) & 1u) << (24 + e);
            }
            const uint32_t lo = __byte_perm(x[0], x[1], 0x7351), hi = __byte_perm(x[2], x[3], 0x7351);      // the bytes with the signs
            const uint32_t even = __byte_perm(lo, hi, 0x5410), odd = __byte_perm(lo, hi, 0x7632);
            next |= (((even >> 4) & 0x08080808u) | (odd & 0x80808080u)) & (next + 0x77777777u);
            w[0] = w[1], w[1] = w[2], w[2] = w[3], w[3] = next;
            if ((i & 3) == 3) {
                *reinterpret_cast<uint4*>(dst + (size_t)((i >> 2) * kTileTokens) * 16) = make_uint4(w[0], w[1], w[2], w[3]);
                if constexpr (K > 0)
#pragma unroll
                    for (int bit = 0; bit < K; ++bit)
                        *reinterpret_cast<uint32_t*>(half + a.plane_off + (size_t)(bit * kTileTokens + t) * (D / 8) + (i & ~3)) = plane[bit];
            }
        }
    }
    *reinterpret_cast<uint16_t*>(half + a.meta_off + (size_t)t * 4) = (uint16_t)smax;
}
template <int D>
SA_D void fill_values(uint8_t* half, const CacheArgs& a, int t, const uint4* src) {
    VecRow<D, false> row(src, t);
    const int g = value_exponent(row.max_bits());
    const float f = pow2i(g);
#pragma unroll 1
    for (int c = 0; c < D / 16; ++c) {
        uint32_t h[8], w[4];
        row.get(2 * c, h);
        row.get(2 * c + 1, h + 4);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            // scaling by 2^g is exact, so adding 1.5 * 2^23 rounds to the nearest integer (ties to even), the low byte of the bits
            const float2 x = half2_bits_to_float2(h[2 * i]), y = half2_bits_to_float2(h[2 * i + 1]);
            const uint32_t lo = __byte_perm(__float_as_uint(__fmaf_rn(x.x, f, 12582912.0f)), __float_as_uint(__fmaf_rn(x.y, f, 12582912.0f)), 0x0040);
            const uint32_t hi = __byte_perm(__float_as_uint(__fmaf_rn(y.x, f, 12582912.0f)), __float_as_uint(__fmaf_rn(y.y, f, 12582912.0f)), 0x0040);
            w[i] = __byte_perm(lo, hi, 0x5410);
        }
        *reinterpret_cast<uint4*>(half + a.v_off + (size_t)(c * kTileTokens + t) * 16) = make_uint4(w[0], w[1], w[2], w[3]);
    }
    *reinterpret_cast<uint16_t*>(half + a.meta_off + (size_t)t * 4 + 2) = (uint16_t)(g & 0xff);
}

template <int D, int MODE, bool HAD>                          // HAD on its own: the rotation needs twice the registers
__global__ void __launch_bounds__(128) fill_kernel(CacheArgs a, const uint16_t* __restrict__ Kin, const uint16_t* __restrict__ Vin,
                                                   const __grid_constant__ FillSeqs seqs) {
    const int lane = threadIdx.x & 31;
    const int64_t unit = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);        // (tile, head, keys or values)
    const int tile = (int)(unit / (2 * a.Hkv)), rest = (int)(unit % (2 * a.Hkv));
    const int head = rest >> 1;
    if (tile >= seqs.tiles[seqs.n]) return;
    int i = 0;                                                                // the sequence: the last one that starts at or before the tile
    for (int j0 = 0; j0 < seqs.n; j0 += 32) {
        const int j = j0 + lane;
        i += __popc(__ballot_sync(0xffffffffu, j < seqs.n && seqs.tiles[j + 1] <= tile));
    }
    const int t = (tile - seqs.tiles[i]) * kTileTokens;                       // first token
    pdl_wait();                                                               // earlier kernels may read this cache or write the inputs
    pdl_launch_dependents();
    uint8_t* block = page_block(a, seqs.b0 + i, t / kPageTokens, head);
    if (!block) return;
    uint8_t* half = block + (size_t)((t % kPageTokens) >> 5) * (a.page_bytes >> 1);
    // the tile's rows, a 16-byte chunk per lane: whole 128-byte lines per load
    constexpr int C = D / 8, R = 32 / C;
    __shared__ uint4 buffers[4][32 * C];
    uint4* src = buffers[threadIdx.x >> 5];
    const int n = seqs.len[i] - t, ch = lane % C;
    const uint4* in = reinterpret_cast<const uint4*>(((rest & 1) ? Vin : Kin) + ((size_t)(seqs.row0[i] + t) * a.Hkv + head) * D) + ch;
    const size_t pitch = (size_t)a.Hkv * C;
    uint4 v[C];
#pragma unroll
    for (int k = 0; k < C; ++k)
        if (k * R + lane / C < n) v[k] = __ldg(in + (size_t)(k * R + lane / C) * pitch);
#pragma unroll
    for (int k = 0; k < C; ++k) {
        const int row = k * R + lane / C;
        if (row < n) src[row * C + (ch ^ (row & 7))] = v[k];
    }
    __syncwarp();
    if (lane >= n) return;
    if constexpr (MODE == 16) {                                               // unquantised: 16-byte chunks of 8 elements
        uint8_t* dst = half + ((rest & 1) ? a.v_off : a.kcode_off);
#pragma unroll
        for (int k = 0; k < D / 8; ++k) *reinterpret_cast<uint4*>(dst + (size_t)(k * kTileTokens + lane) * 16) = src[lane * C + (k ^ (lane & 7))];
    } else {
        if (rest & 1) fill_values<D>(half, a, lane, src);
        else fill_keys<D, MODE, HAD>(half, a, lane, src);
    }
}

// sa_debug_unpack
template <int D, bool NIB>
__global__ void __launch_bounds__(128) unpack_kernel(CacheArgs a, int b, int T, uint8_t xor_mask, int planes, uint8_t* __restrict__ codes,
                                                     uint16_t* __restrict__ scales, int8_t* __restrict__ vhat,
                                                     int8_t* __restrict__ g) {
    constexpr int EPL = D / 32;
    const int lane = threadIdx.x & 31;
    const int64_t v = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
    if (v >= (int64_t)T * a.Hkv) return;
    const int tt = (int)(v / a.Hkv), h = (int)(v % a.Hkv);
    const uint8_t* block = page_block(a, b, tt / kPageTokens, h);
    if (!block) return;
    block += (size_t)((tt % kPageTokens) >> 5) * (a.page_bytes >> 1);      // the token's half of the page
    const int t = tt & 31;
    const int m = lane * EPL;
    if (codes) {
        uint8_t c[EPL];
        if (!NIB) {
            const uint8_t* src = block + a.kcode_off + ((size_t)(m >> 4) * kTileTokens + t) * 16 + (m & 15);
#pragma unroll
            for (int i = 0; i < EPL; ++i) c[i] = xor_mask ? canon_byte(src[i]) : src[i];   // power-of-two codes / INT8 stored as is
        } else {
            const uint8_t* src = block + a.kcode_off + ((size_t)(m >> 5) * kTileTokens + t) * 16 + ((m & 31) >> 1);
#pragma unroll
            for (int i = 0; i < EPL / 2; ++i) {
                c[2 * i] = (uint8_t)((src[i] << 4) ^ 0x70);
                c[2 * i + 1] = (uint8_t)((src[i] & 0xf0) ^ 0x70);
            }
            // dense planar container: the canonical mantissa is left-aligned in the low nibble
            for (int bit = 0; bit < planes; ++bit) {
                const uint8_t* pl = block + a.plane_off + ((size_t)bit * kTileTokens + t) * (D / 8);
#pragma unroll
                for (int i = 0; i < EPL; ++i) c[i] |= (uint8_t)(((pl[(m + i) >> 3] >> ((m + i) & 7)) & 1u) << (4 - planes + bit));
            }
        }
        store_bytes<EPL>(codes + (size_t)v * D + m, c);
    }
    if (vhat) {
        const uint8_t* src = block + a.v_off + ((size_t)(m >> 4) * kTileTokens + t) * 16 + (m & 15);
        uint8_t c[EPL];
#pragma unroll
        for (int i = 0; i < EPL; ++i) c[i] = src[i];
        store_bytes<EPL>(reinterpret_cast<uint8_t*>(vhat) + (size_t)v * D + m, c);
    }
    if (lane == 0) {
        const uint32_t meta = *reinterpret_cast<const uint32_t*>(block + a.meta_off + (size_t)t * 4);
        if (scales) scales[v] = (uint16_t)(meta & 0xffffu);
        if (g) g[v] = (int8_t)((meta >> 16) & 0xff);
    }
}

static bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }

static sa_status check_cache(const Plan& p, const sa_cache* c, CacheArgs* a) {
    if (!c || !c->pages || !c->page_table || !c->seq_lens) return SA_ERR_INVALID_ARG;
    if (c->batch <= 0 || c->max_pages_per_seq <= 0 || c->n_pages <= 0) return SA_ERR_INVALID_ARG;
    if (!aligned(c->pages, p.lay.align) || !aligned(c->page_table, 4) || !aligned(c->seq_lens, 4))
        return SA_ERR_ALIGNMENT;
    a->pages = static_cast<uint8_t*>(c->pages);
    a->page_table = c->page_table;
    a->seq_lens = c->seq_lens;
    a->batch = c->batch;
    a->max_pages = c->max_pages_per_seq;
    a->n_pages = c->n_pages;
    a->Hkv = p.Hkv;
    a->page_bytes = p.lay.page_bytes;
    a->kcode_off = p.lay.kcode_off;
    a->meta_off = p.lay.meta_off;
    a->v_off = p.lay.v_off;
    a->plane_off = p.plane_off;
    a->hadamard = p.hadamard ? 1 : 0;
    return SA_OK;
}

static int mode_of(const Plan& p) { return p.fp16 ? 16 : (p.int8 ? 32 : (p.nibble ? 8 + p.k : p.k)); }

#define SA_LAUNCH_CHECK() (cudaGetLastError() == cudaSuccess ? SA_OK : SA_ERR_CUDA)

// Dispatch over (head_dim, storage mode).
#define SA_DISPATCH_D_MODE(p, CALL)                                                     \
    do {                                                                                \
        const int mode_ = mode_of(p);                                                   \
        if ((p).d == 64) {                                                              \
            switch (mode_) {                                                            \
                case 0: CALL(64, 0); break;                                             \
                case 1: CALL(64, 1); break;                                             \
                case 2: CALL(64, 2); break;                                             \
                case 4: CALL(64, 4); break;                                             \
                case 8: CALL(64, 8); break;                                             \
                case 9: CALL(64, 9); break;                                             \
                case 10: CALL(64, 10); break;                                           \
                case 32: CALL(64, 32); break;                                           \
                default: CALL(64, 16); break;                                           \
            }                                                                           \
        } else {                                                                        \
            switch (mode_) {                                                            \
                case 0: CALL(128, 0); break;                                            \
                case 1: CALL(128, 1); break;                                            \
                case 2: CALL(128, 2); break;                                            \
                case 4: CALL(128, 4); break;                                            \
                case 8: CALL(128, 8); break;                                            \
                case 9: CALL(128, 9); break;                                            \
                case 10: CALL(128, 10); break;                                          \
                case 32: CALL(128, 32); break;                                          \
                default: CALL(128, 16); break;                                          \
            }                                                                           \
        }                                                                               \
    } while (0)

}  // namespace sa

using namespace sa;

extern "C" {

sa_status sa_encode_keys(const sa_config* cfg, const uint16_t* K, int64_t n, uint8_t* codes,
                         uint16_t* scales, sa_stream stream) {
    Plan p;
    sa_status st = make_plan(cfg, &p);
    if (st != SA_OK) return st;
    if (p.fp16) return SA_ERR_UNSUPPORTED;
    if (!K || !codes || !scales || n < 0) return SA_ERR_INVALID_ARG;
    if (!aligned(K, 16) || !aligned(codes, 16) || !aligned(scales, 2)) return SA_ERR_ALIGNMENT;
    const int64_t n_vec = n * p.Hkv;
    if (n_vec == 0) return SA_OK;
    if ((n_vec + 3) / 4 > 0x7fffffffLL) return SA_ERR_CAPACITY;
    const unsigned grid = (unsigned)((n_vec + 3) / 4);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int had = p.hadamard ? 1 : 0;
#define CALL(D, KK) encode_keys_kernel<D, KK><<<grid, 128, 0, s>>>(K, n_vec, codes, scales, had)
    if (p.int8) {
        if (p.d == 64) CALL(64, 8);
        else CALL(128, 8);
    } else if (p.d == 64) {
        switch (p.k) { case 0: CALL(64, 0); break; case 1: CALL(64, 1); break; case 2: CALL(64, 2); break; default: CALL(64, 4); }
    } else {
        switch (p.k) { case 0: CALL(128, 0); break; case 1: CALL(128, 1); break; case 2: CALL(128, 2); break; default: CALL(128, 4); }
    }
#undef CALL
    return SA_LAUNCH_CHECK();
}

sa_status sa_quantise_query(const sa_config* cfg, const uint16_t* Q, int batch, int8_t* q_hat,
                            float* delta, sa_stream stream) {
    Plan p;
    sa_status st = make_plan(cfg, &p);
    if (st != SA_OK) return st;
    if (!Q || !q_hat || !delta || batch < 0) return SA_ERR_INVALID_ARG;
    if (!aligned(Q, 16) || !aligned(q_hat, 16) || !aligned(delta, 4)) return SA_ERR_ALIGNMENT;
    const int64_t n_vec = (int64_t)batch * p.Hq;
    if (n_vec == 0) return SA_OK;
    const unsigned grid = (unsigned)((n_vec + 3) / 4);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int had = (p.hadamard && !p.fp16) ? 1 : 0;
    if (p.d == 64) quantise_query_kernel<64><<<grid, 128, 0, s>>>(Q, n_vec, q_hat, delta, had);
    else quantise_query_kernel<128><<<grid, 128, 0, s>>>(Q, n_vec, q_hat, delta, had);
    return SA_LAUNCH_CHECK();
}

sa_status sa_quantise_values(const sa_config* cfg, const uint16_t* V, int64_t n, int8_t* v_hat,
                             int8_t* g, sa_stream stream) {
    Plan p;
    sa_status st = make_plan(cfg, &p);
    if (st != SA_OK) return st;
    if (!V || !v_hat || !g || n < 0) return SA_ERR_INVALID_ARG;
    if (!aligned(V, 16) || !aligned(v_hat, 16)) return SA_ERR_ALIGNMENT;
    const int64_t n_vec = n * p.Hkv;
    if (n_vec == 0) return SA_OK;
    if ((n_vec + 3) / 4 > 0x7fffffffLL) return SA_ERR_CAPACITY;
    const unsigned grid = (unsigned)((n_vec + 3) / 4);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if (p.d == 64) quantise_values_kernel<64><<<grid, 128, 0, s>>>(V, n_vec, v_hat, g);
    else quantise_values_kernel<128><<<grid, 128, 0, s>>>(V, n_vec, v_hat, g);
    return SA_LAUNCH_CHECK();
}

sa_status sa_append_kv(const sa_config* cfg, const sa_cache* cache, const uint16_t* K_new,
                       const uint16_t* V_new, int bump_lens, sa_stream stream) {
    Plan p;
    sa_status st = make_plan(cfg, &p);
    if (st != SA_OK) return st;
    CacheArgs a;
    st = check_cache(p, cache, &a);
    if (st != SA_OK) return st;
    if (!K_new || !V_new) return SA_ERR_INVALID_ARG;
    if (!aligned(K_new, 16) || !aligned(V_new, 16)) return SA_ERR_ALIGNMENT;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
#define CALL(D, M) (void)launch_pdl(append_kernel<D, M>, dim3(a.batch), dim3(128), 0, s, a, K_new, V_new, bump_lens)
    SA_DISPATCH_D_MODE(p, CALL);
#undef CALL
    return SA_LAUNCH_CHECK();
}

sa_status sa_fill_kv(const sa_config* cfg, const sa_cache* cache, const uint16_t* K, const uint16_t* V,
                     const int64_t* cu_lens_host, sa_stream stream) {
    Plan p;
    sa_status st = make_plan(cfg, &p);
    if (st != SA_OK) return st;
    CacheArgs a;
    st = check_cache(p, cache, &a);
    if (st != SA_OK) return st;
    if (!cu_lens_host) return SA_ERR_INVALID_ARG;
    for (int b = 0; b < a.batch; ++b) {
        const int64_t T = cu_lens_host[b + 1] - cu_lens_host[b];
        if (T < 0 || cu_lens_host[b] < 0) return SA_ERR_INVALID_ARG;
        if (T > (int64_t)a.max_pages * kPageTokens) return SA_ERR_CAPACITY;
    }
    if (cu_lens_host[a.batch] == cu_lens_host[0]) return SA_OK;   // nothing to write
    if (!K || !V) return SA_ERR_INVALID_ARG;
    if (!aligned(K, 16) || !aligned(V, 16)) return SA_ERR_ALIGNMENT;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    for (int b0 = 0; b0 < a.batch; b0 += kFillBatch) {
        FillSeqs seqs{};
        seqs.b0 = b0;
        seqs.n = a.batch - b0 < kFillBatch ? a.batch - b0 : kFillBatch;
        for (int i = 0; i < seqs.n; ++i) {
            seqs.row0[i] = cu_lens_host[b0 + i];
            seqs.len[i] = (int)(cu_lens_host[b0 + i + 1] - cu_lens_host[b0 + i]);
            seqs.tiles[i + 1] = seqs.tiles[i] + (seqs.len[i] + kTileTokens - 1) / kTileTokens;
        }
        const int64_t units = (int64_t)seqs.tiles[seqs.n] * 2 * a.Hkv;
        if (units == 0) continue;
        if ((units + 3) / 4 > 0x7fffffffLL) return SA_ERR_CAPACITY;
        const unsigned grid = (unsigned)((units + 3) / 4);
#define CALL(D, M)                                                                               \
    if (M != 16 && a.hadamard) (void)launch_pdl(fill_kernel<D, M, M != 16>, dim3(grid), dim3(128), 0, s, a, K, V, seqs);        \
    else (void)launch_pdl(fill_kernel<D, M, false>, dim3(grid), dim3(128), 0, s, a, K, V, seqs)
        SA_DISPATCH_D_MODE(p, CALL);
#undef CALL
        if (cudaGetLastError() != cudaSuccess) return SA_ERR_CUDA;
    }
    return SA_OK;
}

sa_status sa_debug_unpack(const sa_config* cfg, const sa_cache* cache, int b, int n_tokens,
                          uint8_t* codes, uint16_t* scales, int8_t* v_hat, int8_t* g, sa_stream stream) {
    Plan p;
    sa_status st = make_plan(cfg, &p);
    if (st != SA_OK) return st;
    if (p.fp16) return SA_ERR_UNSUPPORTED;
    CacheArgs a;
    st = check_cache(p, cache, &a);
    if (st != SA_OK) return st;
    if (b < 0 || b >= a.batch || n_tokens < 0) return SA_ERR_INVALID_ARG;
    if (n_tokens > a.max_pages * kPageTokens) return SA_ERR_CAPACITY;
    if ((codes && !aligned(codes, 16)) || (v_hat && !aligned(v_hat, 16))) return SA_ERR_ALIGNMENT;
    if (n_tokens == 0) return SA_OK;
    const unsigned grid = (unsigned)(((int64_t)n_tokens * a.Hkv + 3) / 4);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const uint8_t xm = p.int8 ? 0x00 : 0x70;
    const int pl = p.nibble ? p.k : 0;                         // mantissa bit planes of the dense planar container
    if (p.d == 64) {
        if (p.nibble) unpack_kernel<64, true><<<grid, 128, 0, s>>>(a, b, n_tokens, xm, pl, codes, scales, v_hat, g);
        else unpack_kernel<64, false><<<grid, 128, 0, s>>>(a, b, n_tokens, xm, pl, codes, scales, v_hat, g);
    } else {
        if (p.nibble) unpack_kernel<128, true><<<grid, 128, 0, s>>>(a, b, n_tokens, xm, pl, codes, scales, v_hat, g);
        else unpack_kernel<128, false><<<grid, 128, 0, s>>>(a, b, n_tokens, xm, pl, codes, scales, v_hat, g);
    }
    return SA_LAUNCH_CHECK();
}

}  // extern "C"
