// Shared declarations of the CUDA library: host-side plan/validation helpers and the small
// exact-arithmetic device functions used by more than one kernel.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>
#include <atomic>

#include "../../include/sa.h"

#define SA_HD __host__ __device__ __forceinline__
#define SA_D __device__ __forceinline__

namespace sa {

constexpr int kPageTokens = 64;
constexpr int kTileTokens = 32;           // a page block is two halves of 32 tokens, each laid out like one staged tile
// Bytes of one half of a (page, KV head) block: code chunks, mantissa bit planes (dense planar container),
// metadata, value chunks.  kb: mantissa bits (8 for the INT8 comparison code); nib: sub-byte container.
// The page plan (make_plan) and the kernels' stage plans are both checked against it.
constexpr int half_block_bytes(int d, int kb, bool nib) {
    return kTileTokens * (nib ? d / 2 : d) + ((nib && kb > 0) ? kb * kTileTokens * (d / 8) : 0) + kTileTokens * 4 + kTileTokens * d;
}
constexpr int half_block_bytes_fp16(int d) { return 2 * kTileTokens * d * 2; }
constexpr int kNumSMsB200 = 148;          // the split plan's SM count where no device can be asked (see sm_count())
constexpr int kEmax = 6;                  // largest exponent of the 3-bit field
constexpr int kMNone = -(1 << 29);        // running-maximum value meaning "no key seen yet"

// Warps per block, resident blocks per SM and stage buffers per warp of a decode kernel (the kernels' launch bounds and
// shared-memory plans are sized for exactly this, and the split plan counts on it).
struct KernelShape {
    int warps, blocks_per_sm, stages;
};
// Matrix kernels (sa_decode_mma.cuh).  kb: mantissa bits, 8 for INT8.
constexpr KernelShape mma_shape(int d, int kb) {
    return d == 128 ? KernelShape{6, 2, 2} : (kb == 1 || kb == 2) ? KernelShape{4, 4, 2} : KernelShape{8, 2, 2};
}
// ... over the binary16 cache (tiles of 8 and 16 KB).
constexpr KernelShape fp16_shape(int d) { return d == 128 ? KernelShape{6, 2, 1} : KernelShape{5, 2, 2}; }
// The kernel of one block per SM (sa_decode_stream.cuh).
constexpr KernelShape stream_shape(int d, bool fp16) {
    return fp16 ? KernelShape{12, 1, d == 128 ? 1 : 2} : d == 128 ? KernelShape{12, 1, 2} : KernelShape{16, 1, 2};
}
SA_HD constexpr int stream_unit_cost(int d) { return d == 128 ? 14 : 32; }     // what a block pays for going on to another unit, in tiles
SA_HD constexpr int stream_merge_cost(int d) { return d == 128 ? 20 : 30; }    // ... for parts of a unit that other blocks have worked on
// U units of T tiles each on P blocks: parts that every unit is cut into (1: units stay whole), where the busiest block, merges
// included, is then done sooner than with a cut that takes no notice of units (0).
SA_HD int stream_parts(int T, int U, int P, int d) {
    const int unit = stream_unit_cost(d), merge = stream_merge_cost(d), k = P / U < T ? P / U : T, c = (U + P - 1) / P;
    const int cut = (U * (T + unit) + P - 1) / P + merge, whole = c * T + (c - 1) * unit, even = k > 1 ? (T + k - 1) / k + merge : 0x7fffffff;
    return (whole < even ? whole : even) > cut ? 0 : even < whole ? k : 1;
}
constexpr int kClusterMost = 8;           // blocks of a thread-block cluster
// ... of the matrix kernels where the splits of a sequence form a cluster.  (fp16: fp16_shape.)
constexpr KernelShape cluster_shape(int d) { return d == 128 ? KernelShape{6, 2, 2} : KernelShape{8, 2, 2}; }
// Shift-and-add kernels (sa_decode_kernel.cuh): one stage buffer per warp where a second one would cost resident warps
// (d = 128, where a tile is 8 KB, and PoT-M4 with its 32 KB table of query multiples).
constexpr KernelShape shift_shape(int d, int kb) {
    const int ns = (d == 128 || kb == 4) ? 1 : 2;
    return (kb == 1 || kb == 2) ? KernelShape{4, 4, ns}
           : (d == 64)          ? KernelShape{10, 2, ns}
           : (kb == 4)          ? KernelShape{8, 2, ns}
                                : KernelShape{4, 5, ns};
}

// ---------------------------------------------------------------------------------------------
// Host-side description of a validated configuration.
// ---------------------------------------------------------------------------------------------
struct Plan {
    int d, Hq, Hkv, G, k;     // k = mantissa bits (0 for SA_KV_FP16)
    bool mulshift;            // SA_FLAG_SHIFT_BY_MULTIPLY: the scores' shifts run on the integer multiplier
    bool addalu;              // SA_FLAG_ADD_ON_ALU: sign flips and adds as logic/add instructions, no multiply-add
    bool shiftadd;            // SA_FLAG_SHIFT_ADD: shifts, and sign flip and add as one multiply-add by +1 / -1
    bool fp16, nibble, hadamard, int8;   // nibble: 4-bit sign/exponent codes (PoT-4 nibble container, or with k = 1, 2
                                         // the dense planar container); int8: the uniform INT8 comparison code
    int F;                    // head-room actually used
    int f_extra;              // F - (6 + k): applied as one final left shift of the INT32 sum
    sa_layout lay;
    size_t plane_off;         // dense planar container: offset of the mantissa bit planes inside a block
    KernelShape shape;        // of the decode kernel that serves this configuration
    bool matrix;              // that kernel is the one of sa_decode_mma.cuh
};

// Does something once for every device (an attribute of a kernel belongs to a device's context): set() is called until it has
// returned true for the device, by several threads at once if they come together, and for devices beyond 63 each time.
struct OncePerDevice {
    std::atomic<uint64_t> done{0};
    template <typename Set>
    bool operator()(int dev, Set set) {
        const uint64_t bit = dev >= 0 && dev < 64 ? 1ull << dev : 0ull;
        if (done.load(std::memory_order_acquire) & bit) return true;
        if (!set()) return false;
        done.fetch_or(bit, std::memory_order_release);
        return true;
    }
};

sa_status make_plan(const sa_config* cfg, Plan* out);
// Streaming multiprocessors of the current device (cudaDevAttrMultiProcessorCount, asked once per device; 148,
// a B200, where no device answers, so that the size queries also work on a machine without a GPU).
int sm_count();
// Number of splits of the key axis for a cache of this shape, and queries handled per block.  cluster (matrix kernel): the
// splits form one thread-block cluster.  stream: the blocks of the kernel of one block per SM where that one serves the call
// (n_splits then only says how much of the workspace it needs), else 0; null: not asked for.  fine: that kernel's form (DecodeArgs).
void split_plan(const Plan& p, int batch, int max_pages, int* n_splits, int* gt, bool* cluster = nullptr, int* stream = nullptr,
                bool* fine = nullptr);

// ---------------------------------------------------------------------------------------------
// Exact helpers (usable on host for unit tests of the arithmetic, and on device).
// ---------------------------------------------------------------------------------------------

// Byte container: physical byte of a canonical code byte (sign << 7 | e << 4 | mantissa << (4 - k)):
//   sign << 7 | mantissa field << 3 | g,   g = 7 - e for a non-zero element, 0 for the zero code.
// The exponent field sits in the low bits (g - 1 is the shift amount), the mantissa field at bits
// 3 .. 6 (times 8 it is the byte offset of a table entry), and zeroed memory reads as zero codes.
SA_HD uint8_t phys_byte(uint8_t canon) {
    return (uint8_t)((canon & 0x80u) | ((canon & 0x0fu) << 3) | (((canon >> 4) & 7u) ^ 7u));
}
SA_HD uint8_t canon_byte(uint8_t phys) {
    return (uint8_t)((phys & 0x80u) | (((phys & 7u) ^ 7u) << 4) | ((phys >> 3) & 0x0fu));
}

// Normalise a non-zero binary16 magnitude (15 bits) to M * 2^X with M in [1024, 2047].
SA_HD void half_normalise(uint32_t mag_bits, int* M, int* X) {
    const int ex = (int)(mag_bits >> 10);
    const int man = (int)(mag_bits & 0x3ff);
    if (ex != 0) {
        *M = 1024 + man;
        *X = ex - 25;
    } else {
#ifdef __CUDA_ARCH__
        const int sh = __clz(man) - 21;
#else
        int sh = 0;
        while (((man << sh) & 0x400) == 0) ++sh;
#endif
        *M = man << sh;
        *X = -24 - sh;
    }
}

SA_HD uint32_t float_bits(float x) {
#ifdef __CUDA_ARCH__
    return __float_as_uint(x);
#else
    uint32_t u;
    memcpy(&u, &x, 4);
    return u;
#endif
}
// A key vector's scale (binary16 bits of its largest magnitude) as the encoder uses it.
struct KeyScale {
    uint32_t M, MM;           // s = M * 2^X with M in [1024, 2047]; M^2
    float inv;                // 1 / s (0 for an all-zero vector)
};
SA_HD KeyScale key_scale(uint32_t s_bits) {
    const float s = __half2float(__ushort_as_half((unsigned short)(s_bits & 0x7fffu)));      // exact, normalised
    KeyScale k;
    k.M = ((float_bits(s) >> 13) & 0x3ffu) | 0x400u;
    k.MM = k.M * k.M;
    k.inv = s > 0.0f ? 1.0f / s : 0.0f;
    return k;
}
// Code of one key element (section II-A, II-D), `a` the element's binary16 value (its sign does not matter), K the number of
// mantissa bits, as the magnitude's place on the grid: g 2^K + j (g = 7 - e) for the codeword (1 + j/2^K) 2^-e, below 2^K: the
// zero code.
//   u = a/s = rho * 2^-e0 with rho in [1, 2);  j = floor((rho - 1) 2^K);  with n = 2^K + j the
//   neighbours on the grid are n and n + 1 (in units of 2^(-K-e0)), and the upper one is nearer
//   in log2 exactly when rho^2 4^K >= n (n + 1).
// e0 and j are the exponent field and the leading mantissa bits of an FP32 quotient: rho 2^K is a whole number or at least
// 1 / 2047 (relative 2^-16) from one, the quotient is within two units in the last place, so raising it by sixteen (2^-19)
// decides both cases.  The comparison is exact: rho = num / M with num = Ma or 2 Ma, num 2^K < 2^16, and both sides fit 32
// bits (n (n + 1) <= 992, M^2 < 2^22).
SA_HD uint32_t encode_place(int K, float a, const KeyScale& s) {
    const uint32_t rb = float_bits(fabsf(a) * s.inv) + 16u;
    const uint32_t place = rb >> (23 - K);                    // (exponent field, j)
    const uint32_t n = (place & ((1u << K) - 1u)) | (1u << K);
    const uint32_t Ma = ((float_bits(a) >> (13 - K)) & (0x3ffu << K)) | (0x400u << K);       // times 2^K
    const uint32_t num = Ma < s.M << K ? 2u * Ma : Ma;
    const int p = (int)place - (120 << K) + (num * num >= (n * n + n) * s.MM ? 1 : 0);
    return (uint32_t)(p < 0 ? 0 : p);
}
// ... as the canonical byte.
SA_HD uint8_t encode_element_k(int K, uint32_t a_bits, const KeyScale& s) {
    const uint32_t p = encode_place(K, __half2float(__ushort_as_half((unsigned short)a_bits)), s);
    if (p < (1u << K)) return 0x70;
    return (uint8_t)(((a_bits >> 8) & 0x80u) | ((7u - (p >> K)) << 4) | ((p & ((1u << K) - 1u)) << (4 - K)));
}
template <int K>
SA_HD uint8_t encode_element(uint32_t a_bits, uint32_t s_bits) { return encode_element_k(K, a_bits, key_scale(s_bits)); }

// Power-of-two exponent g of the value scale: the largest g with amax * 2^g <= 127
// (section II-E).  amax = M * 2^X, so amax * 2^g <= 127  <=>  M * 2^(X + g + 4) <= 2032.
SA_HD int value_exponent(uint32_t amax_bits) {
    if ((amax_bits & 0x7fffu) == 0) return 0;
    int M, X;
    half_normalise(amax_bits & 0x7fffu, &M, &X);
    return (M <= 2032) ? (-4 - X) : (-5 - X);
}

#ifdef __CUDACC__
// ---------------------------------------------------------------------------------------------
// Device-only helpers.
// ---------------------------------------------------------------------------------------------

// Left shift with the PTX guarantee that amounts >= 32 give 0.  The zero code (e = 7) yields
// the shift amount 6 - 7 = 0xffffffff, so a zero element contributes 0 without a branch.
SA_D uint32_t shl_clamp(uint32_t x, uint32_t n) {
    uint32_t r;
    asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(n));
    return r;
}

// Programmatic dependent launch: a kernel launched with the attribute may start while its
// predecessor in the stream is still draining; it must call pdl_wait() before it touches anything the
// predecessor wrote.  Both are no-ops in a kernel launched the ordinary way.
SA_D void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
SA_D void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

SA_D uint32_t warp_max_u32(uint32_t v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
SA_D float warp_max_f32(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
SA_D float warp_sum_f32(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

SA_D float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Packed FP32 pairs of sm_100, two lanes held in one 64-bit register: a * b + c, a * b, a + b.
using f32x2 = unsigned long long;
SA_D f32x2 ffma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
SA_D f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
SA_D f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
SA_D unsigned long long pack_f32x2(float lo, float hi) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
SA_D void unpack_f32x2(unsigned long long v, float* lo, float* hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(*lo), "=f"(*hi) : "l"(v));
}

// Walsh-Hadamard rotation of one head vector spread over a warp: lane l holds elements
// l*EPL .. l*EPL+EPL-1 in x[].  Sylvester order, butterflies with strides 1, 2, ..., d/2, each
// (a, b) <- (a + b, a - b) in FP32 with one rounding per add (no contraction is possible: there
// is no multiply), then one multiply by 1/sqrt(d) and a round to binary16.  Returns the rotated
// elements as binary16 bit patterns.
template <int EPL>
SA_D void hadamard_warp(float (&x)[EPL], uint32_t (&bits)[EPL], int lane) {
#pragma unroll
    for (int h = 1; h < EPL; h <<= 1) {
#pragma unroll
        for (int i = 0; i < EPL; ++i)
            if ((i & h) == 0) {
                const float a = x[i], b = x[i + h];
                x[i] = __fadd_rn(a, b);
                x[i + h] = __fsub_rn(a, b);
            }
    }
#pragma unroll
    for (int hl = 1; hl < 32; hl <<= 1) {
#pragma unroll
        for (int i = 0; i < EPL; ++i) {
            const float other = __shfl_xor_sync(0xffffffffu, x[i], hl);
            x[i] = (lane & hl) ? __fsub_rn(other, x[i]) : __fadd_rn(x[i], other);
        }
    }
    const float scale = (EPL == 2) ? 0.125f : 0.088388346f;   // 1/sqrt(64), 1/sqrt(128)
#pragma unroll
    for (int i = 0; i < EPL; ++i) bits[i] = __half_as_ushort(__float2half_rn(__fmul_rn(x[i], scale)));
}

// First tile of split s when n_tiles tiles are cut into n_splits slices: floor(n_tiles * s / n_splits) in 32-bit
// unsigned arithmetic (a 64-bit division is a long software routine on the GPU, and this sits on the critical
// path of every block); the host refuses caches with max tiles * splits >= 2^31.
SA_D int split_begin(int n_tiles, int s, int n_splits) {
    return (int)((uint32_t)n_tiles * (uint32_t)s / (uint32_t)n_splits);
}
// 2^e as a float, built from the exponent field; e must lie in [-126, 127].
SA_D float pow2i(int e) { return __int_as_float((e + 127) << 23); }
// 2^e for e <= 0, flushing to 0 below the normal range (used for softmax rescales, which are
// exact power-of-two factors because the running maximum is an integer).
SA_D float pow2i_neg(int e) { return e < -126 ? 0.0f : __int_as_float((e + 127) << 23); }

SA_D float half_bits_to_float(uint32_t b) { return __half2float(__ushort_as_half((unsigned short)b)); }
#endif  // __CUDACC__

#ifdef __CUDACC__
// Launch with programmatic stream serialisation allowed (see pdl_wait above), in clusters of `cluster` blocks along x.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl_cluster(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, unsigned cluster, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args... args) {
    return launch_pdl_cluster(kernel, grid, block, smem, s, 1u, args...);
}
// Opts a kernel in to `bytes` of dynamic shared memory on the current device where that is more than the 48 KB every kernel
// may have; `once` is the kernel's own.  False: the attribute was refused (the runtime's last error says why).
template <typename... KArgs>
inline bool allow_shared(void (*kernel)(KArgs...), int bytes, OncePerDevice& once) {
    int dev = -1;
    if (bytes <= 48 * 1024) return true;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    return once(dev, [&] { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess; });
}
#endif

}  // namespace sa
