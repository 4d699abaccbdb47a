// Quantised lookup tables (Sec. 4.5 and Table 8 of arXiv 2503.15798): the tables are compressed after
// training to the 4-bit and 3-bit NormalFloat types of the QLoRA paper with block-wise absmax scaling,
// which cuts the bytes gathered per token to 25.3 % / 19.5 % of the 16-bit table.  This file holds the
// codebooks, the GPU quantiser that packs a bf16 table into per-id records, and the fused layer that
// gathers a token's packed record and de-quantises inside the weighted sum.
//
// Record of one id (the unit that is gathered; a multiple of 16 bytes, zero padded):
//   NF4: N rows of d/2 bytes -- byte i of a row holds code 2i in its low and code 2i+1 in its high
//        nibble -- then N * d/block float32 scales (the blocks' absolute maxima), row after row.
//   NF3: N rows of d/4 bytes with the two low bits of every code (byte i: codes 4i .. 4i+3, code 4i+k at
//        bits 2k, 2k+1), then N rows of d/8 bytes with the high bits (byte i: codes 8i .. 8i+7, code
//        8i+k at bit k), then N * d/block float16 scales.
// With the paper's blocks (768 for NF4, 128 for NF3) that is 388 bytes per 768 elements and 50 bytes per
// 128 elements: the 25.3 % and 19.5 % of Table 8.  A block never straddles two rows.
#include <cuda_fp16.h>
#include <math.h>
#include <mutex>
#include <string.h>

#include "mole_decode.cuh"

namespace mole {

// ---- codebooks -----------------------------------------------------------------------------------
// k-bit NormalFloat (QLoRA, Sec. 3): quantiles of N(0,1) at evenly spaced probabilities, 2^(k-1) of them
// for the negative half and 2^(k-1) + 1 for the positive half (both counts include the median, so that
// zero is a value of its own), divided by the largest magnitude.  The outermost probability is
// 1 - delta, delta the mean of 1/(2 (2^k - 1)) and 1/(2 2^k).
static double normal_quantile(double prob)
{
    // bisection on the normal CDF written with erfc; the CDF is monotone and 1e-17 wide brackets
    // are far below float32 resolution
    double lo = -12.0, hi = 12.0;
    for (int it = 0; it < 200; ++it) {
        const double mid = 0.5 * (lo + hi);
        const double cdf = 0.5 * erfc(-mid * 0.70710678118654752440);
        if (cdf < prob) lo = mid;
        else hi = mid;
    }
    return 0.5 * (lo + hi);
}

static void build_codebook(int bits, float *out)
{
    const int n = 1 << bits, half = n / 2;
    const double delta = 0.5 * (1.0 / (2.0 * (n - 1)) + 1.0 / (2.0 * n));
    double v[16];
    // positive half: half + 1 probabilities from 1/2 to 1 - delta; index half - 1 is the median (zero)
    for (int i = 0; i <= half; ++i) {
        const double prob = 0.5 + (0.5 - delta) * i / half;
        v[half - 1 + i] = i == 0 ? 0.0 : normal_quantile(prob);
    }
    // negative half: half probabilities from 1/2 down to delta; the median is shared
    for (int i = 1; i < half; ++i) {
        const double prob = 0.5 + (0.5 - delta) * i / (half - 1);
        v[half - 1 - i] = -normal_quantile(prob);
    }
    const double top = v[n - 1] > -v[0] ? v[n - 1] : -v[0];
    for (int i = 0; i < n; ++i) out[i] = static_cast<float>(v[i] / top);
}

struct Codebooks {
    float nf4[16], nf3[8];
};
static const Codebooks &codebooks()
{
    static Codebooks cb;
    static std::once_flag once;
    std::call_once(once, [] {
        build_codebook(4, cb.nf4);
        build_codebook(3, cb.nf3);
    });
    return cb;
}

static int format_bits(int format) { return format == MOLE_LUT_NF4 ? 4 : (format == MOLE_LUT_NF3 ? 3 : 0); }
static int scale_bytes(int format) { return format == MOLE_LUT_NF4 ? 4 : 2; }

static long long record_bytes(int N, int d, int format, int block)
{
    const long long codes = format == MOLE_LUT_NF4 ? static_cast<long long>(N) * d / 2 : static_cast<long long>(N) * (d / 4 + d / 8);
    const long long scales = static_cast<long long>(N) * (d / block) * scale_bytes(format);
    return (codes + scales + 15) / 16 * 16;
}

static int check_format(int N, int d, int format, int block)
{
    if (format != MOLE_LUT_NF4 && format != MOLE_LUT_NF3) return MOLE_ERR_INVALID_ARG;
    if (N < 1 || N > 64 || d < 32 || d % 32 != 0) return MOLE_ERR_UNSUPPORTED_SHAPE;
    if (block < 32 || block % 32 != 0 || d % block != 0) return MOLE_ERR_UNSUPPORTED_SHAPE;
    return MOLE_OK;
}

struct CodebookParam {
    float value[16];
    float mid[15];  // midpoints of adjacent values: a normalised element takes the code = number of midpoints below it
};
static CodebookParam codebook_param(int format)
{
    CodebookParam c;
    memset(&c, 0, sizeof c);
    const int n = 1 << format_bits(format);
    const float *src = format == MOLE_LUT_NF4 ? codebooks().nf4 : codebooks().nf3;
    for (int i = 0; i < n; ++i) c.value[i] = src[i];
    for (int i = 0; i + 1 < n; ++i) c.mid[i] = 0.5f * (src[i] + src[i + 1]);
    for (int i = n - 1; i < 15; ++i) c.mid[i] = INFINITY;
    return c;
}

// ---- quantiser, any block size: one block of threads per id (blocks above 2048 elements) ---------------
// Pass 1: a warp per quantisation block finds the absolute maximum and stores the scale (float32, or the
// float16 rounding of min(max, 65504)).  Pass 2: a thread per 8 consecutive elements divides by the stored
// scale in float32 (IEEE division), counts the midpoints below the quotient and packs the 8 codes.
constexpr int kQuantThreads = 256;

template <int BITS>
__global__ void __launch_bounds__(kQuantThreads) mole_quantize_wide_kernel(const uint4 *__restrict__ src, unsigned char *__restrict__ dst,
                                                                      long long V, int N, int d, int block, long long rec_bytes,
                                                                      const CodebookParam cb)
{
    extern __shared__ float s_scale[];  // [N * d / block] effective scales of this id
    const long long id = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = kQuantThreads / 32;
    const int nblk = d / block, total_blocks = N * nblk;
    const uint4 *row0 = src + id * (static_cast<long long>(N) * d / 8);
    unsigned char *rec = dst + id * rec_bytes;
    const long long code_bytes = BITS == 4 ? static_cast<long long>(N) * d / 2 : static_cast<long long>(N) * (d / 4 + d / 8);
    for (int b = warp; b < total_blocks; b += nwarps) {
        const int j = b / nblk, kb = b % nblk;
        const uint4 *p = row0 + (static_cast<long long>(j) * d + static_cast<long long>(kb) * block) / 8;
        float m = 0.f;
        for (int g = lane; g < block / 8; g += 32) {
            float f[8];
            Elem<__nv_bfloat16>::unpack(__ldg(p + g), f);
#pragma unroll
            for (int i = 0; i < 8; ++i) m = fmaxf(m, fabsf(f[i]));
        }
        m = warp_max(m);
        if (lane == 0) {
            if constexpr (BITS == 4) {
                reinterpret_cast<float *>(rec + code_bytes)[b] = m;
                s_scale[b] = m;
            } else {
                const __half h = __float2half_rn(fminf(m, 65504.f));
                reinterpret_cast<__half *>(rec + code_bytes)[b] = h;
                s_scale[b] = __half2float(h);
            }
        }
    }
    __syncthreads();
    const int groups = N * d / 8;  // groups of 8 consecutive elements
    for (int g = tid; g < groups; g += kQuantThreads) {
        const int j = g / (d / 8), c8 = g % (d / 8);
        const float s = s_scale[j * nblk + (c8 * 8) / block];
        float f[8];
        Elem<__nv_bfloat16>::unpack(__ldg(row0 + g), f);
        uint32_t code[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float y = s > 0.f ? __fdiv_rn(f[i], s) : 0.f;
            uint32_t k = 0;
#pragma unroll
            for (int t = 0; t < (1 << BITS) - 1; ++t) k += y > cb.mid[t] ? 1u : 0u;
            code[i] = k;
        }
        if constexpr (BITS == 4) {
            uint32_t w = 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) w |= code[i] << (4 * i);
            reinterpret_cast<uint32_t *>(rec)[g] = w;  // 4 bytes: codes 8 c8 .. 8 c8 + 7 of row j
        } else {
            uint32_t a = 0, b = 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                a |= (code[i] & 3u) << (2 * i);
                b |= ((code[i] >> 2) & 1u) << i;
            }
            reinterpret_cast<unsigned short *>(rec)[g] = static_cast<unsigned short>(a);                   // low bits, 2 bytes
            rec[static_cast<long long>(N) * (d / 4) + g] = static_cast<unsigned char>(b);                // high bits, 1 byte
        }
    }
    // padding bytes after the scales stay as the caller left them (zero them once after allocation if
    // records are to compare equal byte for byte)
}

// ---- quantiser, blocks of up to 2048 elements: a group of 2 .. 32 lanes per quantisation block ------------
// Bound by memory: a table is read once and a quarter or a fifth of it written.  To stay under that the decision per
// element is made without a division and two elements at a time.  The code of x is the number of codebook midpoints
// below fl(x / s); no bf16 x and no scale s of at most 11 significant bits (a bf16, or the float16 an NF3 scale is)
// has a quotient within a rounding of a midpoint (all mantissa pairs enumerated in tests/test_gpu_quant_tiles.py), so
// fl(x / s) > m is x > s m in exact arithmetic, and for a bf16 x that is x > T, T the product rounded towards minus
// infinity first to float32 and then to bf16.  The midpoints' thresholds are made once per quantisation block and
// searched by bisection with packed bf16 compares.  A lane owns chunks of 16 consecutive elements (one 32-byte load; 8
// bytes of NF4 codes, 4 + 2 of NF3) and keeps them in registers between the maximum and the coding.
// One layer of the 160M shape (618 M elements) to NF3, block 128: 369 us before the bounds below, 345 with them (1486 us with two passes and a division
// and 7 float32 compares per element); what is left is the integer pipe (compares and selects): 78 % busy, and 84 % to NF4 in blocks of 1024,
// at 63 % of the issue slots.
__device__ __forceinline__ uint32_t bf162_bits(__nv_bfloat162 v) { return *reinterpret_cast<const uint32_t *>(&v); }
__device__ __forceinline__ __nv_bfloat162 bits_bf162(uint32_t v) { return *reinterpret_cast<const __nv_bfloat162 *>(&v); }
// 0xffff in each half where x > t
__device__ __forceinline__ uint32_t gt2(uint32_t x, uint32_t t) { return __hgt2_mask(bits_bf162(x), bits_bf162(t)); }
// per bit: m ? a : b
__device__ __forceinline__ uint32_t sel2(uint32_t m, uint32_t a, uint32_t b) { return (a & m) | (b & ~m); }
// s * mid rounded towards minus infinity to float32, then to bf16; in both halves of the word
template <bool NEGATIVE>
__device__ __forceinline__ uint32_t threshold2(float s, float mid)
{
    uint32_t u = __float_as_uint(__fmul_rd(s, mid));
    if (NEGATIVE) u += 0xffffu;
    return __byte_perm(u, u, 0x3232);
}
// masks of the code bits of two elements: m[b] has 0xffff in a half whose code has bit b
template <int BITS>
struct CodeSearch;
template <>
struct CodeSearch<3> {
    uint32_t t[7];
    __device__ __forceinline__ void code(uint32_t x, uint32_t (&m)[3]) const
    {
        m[2] = gt2(x, t[3]);
        m[1] = gt2(x, sel2(m[2], t[5], t[1]));
        m[0] = gt2(x, sel2(m[2], sel2(m[1], t[6], t[4]), sel2(m[1], t[2], t[0])));
    }
};
template <>
struct CodeSearch<4> {
    uint32_t t[15];
    __device__ __forceinline__ void code(uint32_t x, uint32_t (&m)[4]) const
    {
        m[3] = gt2(x, t[7]);
        m[2] = gt2(x, sel2(m[3], t[11], t[3]));
        m[1] = gt2(x, sel2(m[3], sel2(m[2], t[13], t[9]), sel2(m[2], t[5], t[1])));
        m[0] = gt2(x, sel2(m[3], sel2(m[2], sel2(m[1], t[14], t[12]), sel2(m[1], t[10], t[8])),
                           sel2(m[2], sel2(m[1], t[6], t[4]), sel2(m[1], t[2], t[0]))));
    }
};

struct QuantGrid {
    long long rec_bytes;
    uint32_t total;                    // quantisation blocks of the whole table
    uint32_t per_id;                   // ... of one id
    uint32_t code_bytes, low_bytes;    // of a record: all code planes, the NF3 low plane
    int block, group_log2, wide_loads; // elements per block; lanes per block; the table is 32-byte aligned
};

// Six blocks of 128 threads per SM (80 registers; left to itself the compiler takes 93 to 98 and four blocks' worth fit): 24 warps hide
// more of the loads than 16, though values of the dividing branch are spilled (none up to two chunks a lane of NF3 and one of NF4; of four chunks NF3 reloads
// 72 bytes a thread and NF4 236: local memory is 3 % and 7 % of the instructions).  20 000 ids, us: NF3 16 x 768 in blocks of 128 151.0 -> 126.6,
// NF4 16 x 768 in blocks of 768 236.8 -> 196.2, 16 x 2048 in blocks of 1024 564.6 -> 501.0; seven blocks 128.5, 196.4, 499.2, three of 256
// threads 128.6, 202.2, 510.
constexpr int kQuantTileThreads = 128;
template <int BITS, int CPL>
__global__ void __launch_bounds__(kQuantTileThreads, 6) mole_quantize_kernel(const unsigned char *__restrict__ src, unsigned char *__restrict__ dst,
                                                                      const QuantGrid q, const CodebookParam cb)
{
    const int G = 1 << q.group_log2, g = threadIdx.x & (G - 1);
    const uint32_t b_raw = blockIdx.x * (static_cast<uint32_t>(kQuantTileThreads) >> q.group_log2) + (threadIdx.x >> q.group_log2);
    const bool live = b_raw < q.total;
    const uint32_t b = live ? b_raw : q.total - 1;
    const int chunks = q.block >> 4;
    const unsigned char *in = src + static_cast<size_t>(b) * (static_cast<uint32_t>(q.block) * 2u);

    uint32_t x[CPL][8];
#pragma unroll
    for (int i = 0; i < CPL; ++i) {
        const int c = g + (i << q.group_log2);
        if (c < chunks) {
            const unsigned char *p = in + static_cast<uint32_t>(c) * 32u;
            if (q.wide_loads) {
                asm volatile("ld.global.nc.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                             : "=r"(x[i][0]), "=r"(x[i][1]), "=r"(x[i][2]), "=r"(x[i][3]), "=r"(x[i][4]), "=r"(x[i][5]), "=r"(x[i][6]), "=r"(x[i][7])
                             : "l"(p));
            } else {
                const uint4 lo = __ldg(reinterpret_cast<const uint4 *>(p)), hi = __ldg(reinterpret_cast<const uint4 *>(p) + 1);
                x[i][0] = lo.x, x[i][1] = lo.y, x[i][2] = lo.z, x[i][3] = lo.w;
                x[i][4] = hi.x, x[i][5] = hi.y, x[i][6] = hi.z, x[i][7] = hi.w;
            }
        } else {
#pragma unroll
            for (int k = 0; k < 8; ++k) x[i][k] = 0u;
        }
    }
    // the block's absolute maximum (NaNs ignored, as fmaxf does)
    __nv_bfloat162 m2 = bits_bf162(0u);
#pragma unroll
    for (int i = 0; i < CPL; ++i)
#pragma unroll
        for (int k = 0; k < 8; ++k) m2 = __hmax2(m2, __habs2(bits_bf162(x[i][k])));
    float m = fmaxf(__uint_as_float(bf162_bits(m2) << 16), __uint_as_float(bf162_bits(m2) & 0xffff0000u));
    for (int o = G >> 1; o >= 1; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));

    const uint32_t id = b / q.per_id, within = b - id * q.per_id;
    unsigned char *rec = dst + static_cast<size_t>(id) * q.rec_bytes;
    float s = m;
    if constexpr (BITS == 3) {
        const __half h = __float2half_rn(fminf(m, 65504.f));
        s = __half2float(h);
        if (live && g == 0) reinterpret_cast<__half *>(rec + q.code_bytes)[within] = h;
    } else {
        if (live && g == 0) reinterpret_cast<float *>(rec + q.code_bytes)[within] = m;
    }
    CodeSearch<BITS> search;
#pragma unroll
    for (int t = 0; t < (1 << BITS) - 1; ++t)  // zero is value 2^(BITS-1) - 1 of the codebook: the midpoints before it are negative
        search.t[t] = t < (1 << (BITS - 1)) - 1 ? threshold2<true>(s, cb.mid[t]) : threshold2<false>(s, cb.mid[t]);
    const bool plain = s >= 0x1p-100f && s < INFINITY;  // every other block (all zero, infinities, scales near underflow) divides

#pragma unroll
    for (int i = 0; i < CPL; ++i) {
        const int c = g + (i << q.group_log2);
        uint32_t mask[8][BITS];
        if (plain) {
#pragma unroll
            for (int k = 0; k < 8; ++k) search.code(x[i][k], mask[k]);
        } else {
#pragma unroll 1
            for (int k = 0; k < 8; ++k) {
                uint32_t xk = 0;
#pragma unroll
                for (int j = 0; j < 8; ++j) xk = j == k ? x[i][j] : xk;  // (registers have no run-time index)
                uint32_t code[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float f = __uint_as_float(e ? xk & 0xffff0000u : xk << 16);
                    const float y = s > 0.f ? __fdiv_rn(f, s) : 0.f;
                    code[e] = 0;
#pragma unroll
                    for (int t = 0; t < (1 << BITS) - 1; ++t) code[e] += y > cb.mid[t] ? 1u : 0u;
                }
#pragma unroll
                for (int j = 0; j < 8; ++j)
#pragma unroll
                    for (int bit = 0; bit < BITS; ++bit)
                        if (j == k) mask[j][bit] = ((code[0] >> bit) & 1u ? 0xffffu : 0u) | ((code[1] >> bit) & 1u ? 0xffff0000u : 0u);
            }
        }
        // pack: even elements in the low halves, odd ones in the high halves, shifted together at the end
        const bool store = live && c < chunks;
        if constexpr (BITS == 4) {
            uint32_t w[4];  // four elements each: nibbles at bits 0 and 8 of either half
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                uint32_t a = 0;
#pragma unroll
                for (int v = 0; v < 2; ++v)
#pragma unroll
                    for (int bit = 0; bit < 4; ++bit) a |= mask[2 * k + v][bit] & ((1u << (8 * v + bit)) | (1u << (16 + 8 * v + 4 + bit)));
                w[k] = a | (a >> 16);
            }
            const uint2 o = make_uint2(__byte_perm(w[0], w[1], 0x5410), __byte_perm(w[2], w[3], 0x5410));
            if (store) *reinterpret_cast<uint2 *>(rec + within * (static_cast<uint32_t>(q.block) / 2) + static_cast<uint32_t>(c) * 8u) = o;
        } else {
            uint32_t lo[2], hi = 0;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                uint32_t a = 0;
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    a |= mask[4 * k + v][0] & ((1u << (4 * v)) | (1u << (16 + 4 * v + 2)));
                    a |= mask[4 * k + v][1] & ((1u << (4 * v + 1)) | (1u << (16 + 4 * v + 3)));
                    hi |= mask[4 * k + v][2] & ((1u << (8 * k + 2 * v)) | (1u << (16 + 8 * k + 2 * v + 1)));
                }
                lo[k] = a | (a >> 16);
            }
            if (store) {
                *reinterpret_cast<uint32_t *>(rec + within * (static_cast<uint32_t>(q.block) / 4) + static_cast<uint32_t>(c) * 4u) = __byte_perm(lo[0], lo[1], 0x5410);
                *reinterpret_cast<unsigned short *>(rec + q.low_bytes + within * (static_cast<uint32_t>(q.block) / 8) + static_cast<uint32_t>(c) * 2u) =
                    static_cast<unsigned short>(hi | (hi >> 16));
            }
        }
    }
}

// Lanes per quantisation block of `chunks` 16-element chunks (at most 128) and chunks per lane (at most 4): the pair that
// leaves the fewest lanes without a chunk, the one with more chunks per lane among equals (thresholds and the maximum's
// shuffles are paid once per lane).
static void quant_group(int chunks, int *group_log2, int *cpl)
{
    int best = 1 << 30;
    for (int lg = 5; lg >= 0; --lg) {
        const int n = (chunks + (1 << lg) - 1) >> lg;
        if (n > 4) break;
        const int slots = n << lg;
        if (slots <= best) {
            best = slots;
            *group_log2 = lg;
            *cpl = n;
        }
    }
}

typedef void (*QuantizeKernel)(const unsigned char *, unsigned char *, const QuantGrid, const CodebookParam);
template <int BITS>
static QuantizeKernel pick_quantize(int cpl)
{
    switch (cpl) {
        case 1: return mole_quantize_kernel<BITS, 1>;
        case 2: return mole_quantize_kernel<BITS, 2>;
        case 3: return mole_quantize_kernel<BITS, 3>;
        default: return mole_quantize_kernel<BITS, 4>;
    }
}

// ---- the fused layer over packed records: one block per token (see mole_decode.cuh for the structure) ----
struct QDecodeParams {
    const void *hidden, *residual, *row_index, *lut, *w_router, *norm_weight;
    void *out;
    float *gates_out;
    uint32_t *status;
    long long rows, rec_bytes;
    int d, block;
    float norm_eps;
    uint32_t flags, wait_polls;
    float cb[16];
};

__host__ __device__ inline uint32_t qdecode_smem_bytes(int N, int d, long long rec_bytes)
{
    return up128(static_cast<uint32_t>(d) * N * 2) + up128(static_cast<uint32_t>(rec_bytes)) + kDecodeMaxWarps * 64 * 4 +
           kDecodeMaxWarps * 4 + 16 * 4 + 32;
}

// Numerator-weighted sum of a record's de-quantised rows over columns 4 tid .. 4 tid + 3 of every expert; returns the sum of the
// numerators.  rec, cb: the record and the codebook (64-byte aligned) in shared memory; e: lane j holds expert j's numerator
// (0 past the experts).  A code's bits, shifted into place, are or-ed into the codebook's address: one look-up per element is
// what bounds the layer at prefill sizes.  Where a warp's 128 columns lie in one quantisation block, lane j forms numerator times
// scale of expert j once for all of them.
template <int N, int BITS>
__device__ __forceinline__ float dequant_sum(uint32_t rec, uint32_t cb, float e, int d, int block, int tid, float (&a)[4])
{
    const int nblk = d / block, blk = (4 * tid) / block, lane = tid & 31;
    const uint32_t code_bytes = BITS == 4 ? static_cast<uint32_t>(N) * d / 2 : static_cast<uint32_t>(N) * (d / 4 + d / 8);
    auto scale = [&](int j) -> float {
        const uint32_t i = code_bytes + static_cast<uint32_t>(BITS == 4 ? 4 : 2) * static_cast<uint32_t>(j * nblk + blk);
        if constexpr (BITS == 4) return __uint_as_float(lds32(rec + i));
        const unsigned short hb = static_cast<unsigned short>(lds16(rec + i));
        return __half2float(*reinterpret_cast<const __half *>(&hb));
    };
    const bool uniform = block % 128 == 0;
    float own = e;
    if (uniform) own = e * scale(lane < N ? lane : 0);
    const float esum = warp_sum(e);
    a[0] = a[1] = a[2] = a[3] = 0.f;
    uint32_t low = rec + static_cast<uint32_t>(BITS == 4 ? 2 * tid : tid), high = rec + static_cast<uint32_t>(N) * (d / 4) + (tid >> 1);
    const uint32_t low_step = static_cast<uint32_t>(BITS == 4 ? d / 2 : d / 4), high_step = static_cast<uint32_t>(d / 8);
    const int high_shift = 4 * (tid & 1);
#pragma unroll
    for (int j = 0; j < N; ++j, low += low_step, high += high_step) {
        float gs = __shfl_sync(0xffffffffu, own, j);
        if (!uniform) gs *= scale(j);
        uint32_t c0, c1, c2, c3;  // addresses of the four values
        if constexpr (BITS == 4) {
            const uint32_t c = lds16(low);
            c0 = ((c << 2) & 0x3cu) | cb, c1 = ((c >> 2) & 0x3cu) | cb, c2 = ((c >> 6) & 0x3cu) | cb, c3 = ((c >> 10) & 0x3cu) | cb;
        } else {
            uint32_t x, y;
            asm volatile("ld.shared.u8 %0, [%1];" : "=r"(x) : "r"(low));
            asm volatile("ld.shared.u8 %0, [%1];" : "=r"(y) : "r"(high));
            y >>= high_shift;
            c0 = ((x << 2) & 0xcu) | ((y << 4) & 0x10u) | cb, c1 = (x & 0xcu) | ((y << 3) & 0x10u) | cb;
            c2 = ((x >> 2) & 0xcu) | ((y << 2) & 0x10u) | cb, c3 = ((x >> 4) & 0xcu) | ((y << 1) & 0x10u) | cb;
        }
        a[0] = fmaf(gs, __uint_as_float(lds32(c0)), a[0]);
        a[1] = fmaf(gs, __uint_as_float(lds32(c1)), a[1]);
        a[2] = fmaf(gs, __uint_as_float(lds32(c2)), a[2]);
        a[3] = fmaf(gs, __uint_as_float(lds32(c3)), a[3]);
    }
    return esum;
}
// residual + sum / esum, one rounding
__device__ __forceinline__ uint2 add_residual4(const float (&a)[4], float inv, uint2 res)
{
    const __nv_bfloat162 lo = __floats2bfloat162_rn(fmaf(a[0], inv, bf16_bits_to_float(res.x & 0xffffu)), fmaf(a[1], inv, __uint_as_float(res.x & 0xffff0000u)));
    const __nv_bfloat162 hi = __floats2bfloat162_rn(fmaf(a[2], inv, bf16_bits_to_float(res.y & 0xffffu)), fmaf(a[3], inv, __uint_as_float(res.y & 0xffff0000u)));
    return make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
}

template <int N, int BITS, int NORM>
__global__ void __launch_bounds__(kDecodeMaxThreads) mole_qdecode_kernel(const QDecodeParams p)
{
    using E = Elem<__nv_bfloat16>;
    constexpr int VEC = 8;
    constexpr int NV = N < VEC ? N : VEC;
    constexpr int QL = N >= VEC ? N / VEC : 1;
    constexpr int CPV = N >= VEC ? 1 : VEC / N;
    constexpr int R = N / 2;
    extern __shared__ __align__(128) unsigned char smem[];

    pdl_enter(p.flags);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int T = blockDim.x, nwarps = T >> 5, d = p.d;
    const long long t = blockIdx.x;
    const uint32_t wr_bytes = static_cast<uint32_t>(d) * N * 2, rec_bytes = static_cast<uint32_t>(p.rec_bytes);
    unsigned char *rec = smem + up128(wr_bytes);
    float *partial = reinterpret_cast<float *>(rec + up128(rec_bytes));
    float *scratch = partial + kDecodeMaxWarps * 64;
    float *cbs = scratch + kDecodeMaxWarps;
    uint64_t *bar = reinterpret_cast<uint64_t *>(cbs + 16);  // [0]: router matrix, [1]: the token's record

    const long long id = (p.flags & MOLE_FLAG_IDS_INT64) ? __ldg(static_cast<const long long *>(p.row_index) + t)
                                                         : static_cast<long long>(__ldg(static_cast<const int *>(p.row_index) + t));
    const bool valid = id >= 0 && id < p.rows;
    if (tid == 0) {
        mbar_init(bar, 1);
        mbar_init(bar + 1, 1);
        mbar_init_fence();
        mbar_expect_tx(bar, wr_bytes);
        bulk_g2s(smem, p.w_router, wr_bytes, bar);
        mbar_expect_tx(bar + 1, rec_bytes);
        bulk_g2s(rec, static_cast<const unsigned char *>(p.lut) + static_cast<size_t>(valid ? id : 0) * rec_bytes, rec_bytes, bar + 1);
    }
    if (tid < 16) cbs[tid] = p.cb[tid];
    __syncthreads();

    pdl_wait();  // the kernel before may have written the norm's scale, too
    const unsigned char *hrow = static_cast<const unsigned char *>(p.hidden) + static_cast<size_t>(t) * d * 2;
    unsigned short hs[R * CPV];
    uint32_t nw[NORM ? R * CPV : 1];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int cc = 0; cc < CPV; ++cc) {
            const int u = tid + r * T;
            const int col = N >= VEC ? u / QL : u * CPV + cc;
            hs[r * CPV + cc] = ldcg_u16(hrow + 2 * col);
            if constexpr (NORM) nw[r * CPV + cc] = ld_scale_u16(static_cast<const unsigned short *>(p.norm_weight) + col);
        }
    const uint2 hown = ldcg_v2(hrow + static_cast<size_t>(tid) * 8);
    uint2 res = hown;
    if (p.residual) res = ldcg_v2(static_cast<const unsigned char *>(p.residual) + static_cast<size_t>(t) * d * 2 + static_cast<size_t>(tid) * 8);

    if constexpr (NORM) {
        const float x0 = bf16_bits_to_float(hown.x & 0xffffu), x1 = __uint_as_float(hown.x & 0xffff0000u);
        const float x2 = bf16_bits_to_float(hown.y & 0xffffu), x3 = __uint_as_float(hown.y & 0xffff0000u);
        float ss = fmaf(x3, x3, fmaf(x2, x2, fmaf(x1, x1, x0 * x0)));
        ss = warp_sum(ss);
        if (lane == 0) scratch[warp] = ss;
        __syncthreads();
        float total = 0.f;
        for (int w = 0; w < nwarps; ++w) total += scratch[w];
        const float rinv = 1.0f / sqrtf(total / static_cast<float>(d) + p.norm_eps);
#pragma unroll
        for (int i = 0; i < R * CPV; ++i) hs[i] = float_to_bf16_bits((bf16_bits_to_float(hs[i]) * rinv) * bf16_bits_to_float(nw[i]));
    }

    // bounded waits for the two bulk copies; after a failure the block computes on whatever its shared
    // memory holds (every address stays inside it and inside its own output row) and says so
    bool timed_out = false;
#pragma unroll
    for (int which = 0; which < 2; ++which) {
        bool ok = false;
        for (uint32_t i = 0; i < p.wait_polls && !ok; ++i) {
            ok = mbar_try_wait(bar + which, 0);
            if (!ok && i > 64) __nanosleep(64);
        }
        if (!ok) {
            timed_out = true;
            for (uint32_t i = 0; i < kDrainPolls && !ok; ++i) {
                ok = mbar_try_wait(bar + which, 0);
                if (!ok) __nanosleep(64);
            }
        }
    }
    if (timed_out && tid == 0 && p.status) atomicOr(p.status, MOLE_STATUS_TIMEOUT);

    float acc[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) acc[i] = 0.f;
    const uint32_t wbase = smem_u32(smem);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const uint4 wv = lds128(wbase + 16u * static_cast<uint32_t>(tid + r * T));
#pragma unroll
        for (int e = 0; e < VEC; ++e) E::fma_elem(acc[e % NV], wv, e, hs[r * CPV + e / NV]);
    }
    int base = 0;
    lane_reduce_scatter<NV, NV, 16, QL>(acc, lane, base);
    partial[warp * N + (N >= VEC ? (lane % QL) * VEC : 0) + base] = acc[0];
    __syncthreads();

    const float e = softmax_numerator<N>(partial, nwarps, lane);

    // ---- weighted sum over the de-quantised rows: value = codebook[code] * scale of its block ----
    float a4[4];
    const float esum = dequant_sum<N, BITS>(smem_u32(rec), smem_u32(cbs), e, d, p.block, tid, a4);
    const float inv = __frcp_rn(esum);
    const uint2 o = valid ? add_residual4(a4, inv, res) : res;
    *reinterpret_cast<uint2 *>(static_cast<unsigned char *>(p.out) + static_cast<size_t>(t) * d * 2 + static_cast<size_t>(tid) * 8) = o;
    if (warp == 0) {
        if (p.gates_out && lane < N) p.gates_out[t * N + lane] = e / esum;
        if (!valid && lane == 0 && p.status) atomicOr(p.status, MOLE_STATUS_BAD_ID);
    }
}

// ---- the fused L-layer step over packed records ------------------------------------------------------------------------
// The arithmetic of mole_qdecode_kernel, in its order (a fused step gives the bits of L single layers), without the launch per
// layer: a block walks its tokens through all L layers with the hidden state in registers and shared memory.  A layer is bound
// by the latency of one token's chain, so what does not depend on it runs ahead: a producer warp streams the packed records
// through a ring of slots (they depend on the id alone), and the threads load the next layer's router matrix from L2 into the
// registers of the one they have just multiplied.
// 160M shape, 12 layers, NF4, 64 tokens: 33.0 us chained -> 19.9 us.
struct QStepParams {
    const void *hidden, *row_index, *lut, *w_router, *norm_weight;
    void *out;
    uint32_t *status;
    long long rows, rec_bytes, lut_stride, wr_stride, norm_stride, M;
    int d, block, L, stages;
    float norm_eps;
    uint32_t flags, wait_polls;
    float cb[16];
};
struct QStepSmem {
    uint32_t slot, off_hid, off_partial, off_scratch, off_cb, off_meta, off_bars, total;
};
__host__ __device__ inline QStepSmem qstep_smem(int d, long long rec_bytes, int stages)
{
    QStepSmem m;
    m.slot = up128(static_cast<uint32_t>(rec_bytes));
    m.off_hid = static_cast<uint32_t>(stages) * m.slot;
    m.off_partial = m.off_hid + up128(static_cast<uint32_t>(d) * 2);
    m.off_cb = m.off_partial + kDecodeMaxWarps * 32 * 4;
    m.off_scratch = m.off_cb + 64;
    m.off_meta = m.off_scratch + kDecodeMaxWarps * 4;
    m.off_bars = m.off_meta + (kMaxStages + 4) * 4;
    m.total = m.off_bars + 2 * kMaxStages * 8;
    return m;
}
__host__ __device__ constexpr int qstep_max_threads(int N) { return N > 16 ? 256 : kDecodeMaxThreads; }

template <int N, int BITS, int NORM>
__global__ void __launch_bounds__(qstep_max_threads(N) + 32) mole_qstep_kernel(const QStepParams p)
{
    using E = Elem<__nv_bfloat16>;
    constexpr int VEC = 8;
    constexpr int NV = N < VEC ? N : VEC;
    constexpr int QL = N >= VEC ? N / VEC : 1;
    constexpr int CPV = N >= VEC ? 1 : VEC / N;
    constexpr int R = N / 2;
    extern __shared__ __align__(128) unsigned char smem[];

    pdl_enter(p.flags);

    const int d = p.d, L = p.L, stages = p.stages, T = d / 4;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = T >> 5;
    const long long G = gridDim.x, b0 = blockIdx.x;
    const int ntok = b0 < p.M ? static_cast<int>((p.M - b0 + G - 1) / G) : 0;
    const uint32_t rec_bytes = static_cast<uint32_t>(p.rec_bytes);
    const QStepSmem m = qstep_smem(d, p.rec_bytes, stages);
    float *partial = reinterpret_cast<float *>(smem + m.off_partial), *scratch = reinterpret_cast<float *>(smem + m.off_scratch);
    volatile int *meta = reinterpret_cast<volatile int *>(smem + m.off_meta);  // [stages] the slot's id is inside the table
    volatile int *dead = meta + kMaxStages;                                    // somebody gave up waiting; [1] chunks issued; [2] raised by nobody
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + m.off_bars), *empty = full + kMaxStages;
    if (tid == 0) {
        for (int st = 0; st < stages; ++st) {
            mbar_init(full + st, 1);
            mbar_init(empty + st, nwarps);
        }
        dead[0] = dead[1] = dead[2] = 0;
        mbar_init_fence();
    }
    if (tid < 16) reinterpret_cast<float *>(smem + m.off_cb)[tid] = p.cb[tid];
    __syncthreads();

    if (tid >= T) {
        // ================= producer warp: the records of this block's (token, layer) items =================
        int batch = -1;
        int st = 0, issued = 0;
        uint32_t ph = 1;
        bool ok = true;
        for (int k = 0; k < ntok && ok; ++k) {
            if ((k & 31) == 0) {  // ids of the next 32 tokens of this block, one per lane
                batch = -1;
                if (k + lane < ntok) batch = __ldg(static_cast<const int *>(p.row_index) + (b0 + static_cast<long long>(k + lane) * G));
            }
            const int id = __shfl_sync(0xffffffffu, batch, k & 31);
            const bool valid = id >= 0 && id < p.rows;
            if (!valid && lane == 0 && p.status) atomicOr(p.status, MOLE_STATUS_BAD_ID);
            for (int l = 0; l < L; ++l) {
                int got = 1;
                if (lane == 0) {
                    if (issued >= stages) got = wait_or_give_up(empty + st, ph, dead, p.wait_polls, true);
                    if (got) {
                        meta[st] = valid ? 1 : 0;
                        mbar_expect_tx(full + st, rec_bytes);  // an id outside the table gathers row 0; its routed term is dropped
                        bulk_g2s(smem + static_cast<size_t>(st) * m.slot,
                                 static_cast<const unsigned char *>(p.lut) + static_cast<size_t>(l) * p.lut_stride + static_cast<size_t>(valid ? id : 0) * rec_bytes, rec_bytes, full + st);
                        dead[1] = issued + 1;
                    } else {
                        report_timeout(dead, p.status);
                    }
                }
                ok = __shfl_sync(0xffffffffu, got, 0) != 0;
                if (!ok) break;
                ++issued;
                if (++st == stages) st = 0, ph ^= 1u;
            }
        }
        if (dead[0]) drain_ring(full, stages, issued);
        return;
    }

    // ================= compute threads =================
    pdl_wait();  // hidden may still be written, and out still read, by the previous kernel
    const uint32_t smem_base = smem_u32(smem), hid_s = smem_base + m.off_hid;
    bool alive = true;
    int st = 0, item = 0;
    uint32_t ph = 0;
    uint4 wreg[R];
    auto load_router = [&](int l) {  // this thread's vectors of layer l's matrix: u = tid + r T
        const uint4 *w = reinterpret_cast<const uint4 *>(static_cast<const unsigned char *>(p.w_router) + static_cast<size_t>(l) * p.wr_stride);
#pragma unroll
        for (int r = 0; r < R; ++r) wreg[r] = ldg_nc_v4(w + tid + r * T);
    };
    if (ntok > 0) load_router(0);
#pragma unroll 1
    for (int k = 0; k < ntok; ++k) {
        const size_t tbyte = static_cast<size_t>(b0 + static_cast<long long>(k) * G) * d * 2 + static_cast<size_t>(tid) * 8;
        uint2 own = ldcg_v2(static_cast<const unsigned char *>(p.hidden) + tbyte);  // columns 4 tid .. 4 tid + 3
#pragma unroll 1
        for (int l = 0; l < L; ++l, ++item) {
            // ---- what the router reads ----
            uint2 read = own;
            if constexpr (NORM) {
                const uint2 wq = __ldg(reinterpret_cast<const uint2 *>(static_cast<const unsigned char *>(p.norm_weight) + static_cast<size_t>(l) * p.norm_stride) + tid);
                const float x0 = bf16_bits_to_float(own.x & 0xffffu), x1 = __uint_as_float(own.x & 0xffff0000u);
                const float x2 = bf16_bits_to_float(own.y & 0xffffu), x3 = __uint_as_float(own.y & 0xffff0000u);
                const float ss = warp_sum(fmaf(x3, x3, fmaf(x2, x2, fmaf(x1, x1, x0 * x0))));
                if (lane == 0) scratch[warp] = ss;
                named_bar_sync(3, T);
                float total = 0.f;
                for (int w = 0; w < nwarps; ++w) total += scratch[w];
                const float rinv = 1.0f / sqrtf(total / static_cast<float>(d) + p.norm_eps);
                const __nv_bfloat162 y01 = __floats2bfloat162_rn((x0 * rinv) * bf16_bits_to_float(wq.x & 0xffffu), (x1 * rinv) * __uint_as_float(wq.x & 0xffff0000u));
                const __nv_bfloat162 y23 = __floats2bfloat162_rn((x2 * rinv) * bf16_bits_to_float(wq.y & 0xffffu), (x3 * rinv) * __uint_as_float(wq.y & 0xffff0000u));
                read = make_uint2(*reinterpret_cast<const uint32_t *>(&y01), *reinterpret_cast<const uint32_t *>(&y23));
            }
            sts64(hid_s + 8u * tid, read);
            named_bar_sync(1, T);

            // ---- router sweep ----
            float acc[NV];
#pragma unroll
            for (int i = 0; i < NV; ++i) acc[i] = 0.f;
            unsigned short hs[R * CPV];
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int cc = 0; cc < CPV; ++cc) {
                    const int u = tid + r * T;
                    hs[r * CPV + cc] = static_cast<unsigned short>(lds16(hid_s + 2u * (N >= VEC ? u / QL : u * CPV + cc)));
                }
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int e = 0; e < VEC; ++e) E::fma_elem(acc[e % NV], wreg[r], e, hs[r * CPV + e / NV]);
            if (l + 1 < L) load_router(l + 1);
            else if (k + 1 < ntok) load_router(0);
            int base = 0;
            lane_reduce_scatter<NV, NV, 16, QL>(acc, lane, base);
            partial[warp * N + (N >= VEC ? (lane % QL) * VEC : 0) + base] = acc[0];
            named_bar_sync(2, T);
            const float e = softmax_numerator<N>(partial, nwarps, lane);

            // ---- weighted sum of the de-quantised record ----
            if (!(alive && mbar_try_wait(full + st, ph))) alive = acquire_slow(full + st, ph, dead, alive, item < dead[1], p.status, lane, p.wait_polls);
            const bool valid = meta[st] != 0;
            float a4[4];
            const float esum = dequant_sum<N, BITS>(smem_base + static_cast<uint32_t>(st) * m.slot, smem_base + m.off_cb, e, d, p.block, tid, a4);
            __syncwarp();
            if (lane == 0) mbar_arrive(empty + st);
            if (++st == stages) st = 0, ph ^= 1u;
            if (valid) own = add_residual4(a4, __frcp_rn(esum), own);
        }
        *reinterpret_cast<uint2 *>(static_cast<unsigned char *>(p.out) + tbyte) = own;
    }
}

typedef void (*QStepKernel)(const QStepParams);
struct QStepVariant {
    QStepKernel fn;
    const char *name;
};
#define MOLE_QS(N, BITS) (norm ? QStepVariant{mole_qstep_kernel<N, BITS, 1>, "qstep<" #N ",nf" #BITS ",1>"} : QStepVariant{mole_qstep_kernel<N, BITS, 0>, "qstep<" #N ",nf" #BITS ",0>"})
static QStepVariant pick_qstep(int N, int bits, bool norm)
{
    switch (N) {
        case 4: return bits == 4 ? MOLE_QS(4, 4) : MOLE_QS(4, 3);
        case 8: return bits == 4 ? MOLE_QS(8, 4) : MOLE_QS(8, 3);
        case 16: return bits == 4 ? MOLE_QS(16, 4) : MOLE_QS(16, 3);
        case 32: return bits == 4 ? MOLE_QS(32, 4) : MOLE_QS(32, 3);
        default: return QStepVariant{nullptr, "none"};
    }
}
// ring depth: enough to keep an item's latency covered, shallow enough that shared memory never limits the resident blocks
static int qstep_stages(int d, long long rec_bytes)
{
    int stages = 4;
    while (stages > 2 && qstep_smem(d, rec_bytes, stages).total > 56u * 1024u) --stages;
    return stages;
}

typedef void (*QDecodeKernel)(const QDecodeParams);
struct QVariant {
    QDecodeKernel fn;
    const char *name;
};
#define MOLE_QV(N, BITS, NORM) QVariant { mole_qdecode_kernel<N, BITS, NORM>, "qdecode<" #N ",nf" #BITS "," #NORM ">" }
static QVariant pick_qdecode(int N, int bits, bool norm)
{
    if (bits == 4) {
        switch (N) {
            case 4: return norm ? MOLE_QV(4, 4, 1) : MOLE_QV(4, 4, 0);
            case 8: return norm ? MOLE_QV(8, 4, 1) : MOLE_QV(8, 4, 0);
            case 16: return norm ? MOLE_QV(16, 4, 1) : MOLE_QV(16, 4, 0);
            case 32: return norm ? MOLE_QV(32, 4, 1) : MOLE_QV(32, 4, 0);
        }
    } else {
        switch (N) {
            case 4: return norm ? MOLE_QV(4, 3, 1) : MOLE_QV(4, 3, 0);
            case 8: return norm ? MOLE_QV(8, 3, 1) : MOLE_QV(8, 3, 0);
            case 16: return norm ? MOLE_QV(16, 3, 1) : MOLE_QV(16, 3, 0);
            case 32: return norm ? MOLE_QV(32, 3, 1) : MOLE_QV(32, 3, 0);
        }
    }
    return QVariant{nullptr, "none"};
}

bool quant_layer_shape_ok(int N, int d, int format, int block)
{
    if (check_format(N, d, format, block) != MOLE_OK) return false;
    if (N != 4 && N != 8 && N != 16 && N != 32) return false;
    if (d % 128 != 0 || d / 4 > kDecodeMaxThreads) return false;
    return qdecode_smem_bytes(N, d, record_bytes(N, d, format, block)) <= 227u * 1024u;
}

int launch_quant_layer(const StepLaunch &a, int format, int block, uint32_t wait_polls)
{
    if (a.M == 0) return MOLE_OK;
    if (a.dtype != MOLE_DTYPE_BF16 || a.L != 1 || !quant_layer_shape_ok(a.N, a.d, format, block)) return MOLE_ERR_UNSUPPORTED_SHAPE;
    if (a.M > 0x7fffffffLL) return MOLE_ERR_TOO_LARGE;
    const QVariant v = pick_qdecode(a.N, format_bits(format), a.norm_weight != nullptr);
    if (!v.fn) return MOLE_ERR_UNSUPPORTED_SHAPE;
    QDecodeParams p;
    p.hidden = a.hidden;
    p.residual = a.residual;
    p.row_index = a.row_index;
    p.lut = a.lut;
    p.w_router = a.w_router;
    p.norm_weight = a.norm_weight;
    p.out = a.out;
    p.gates_out = a.gates_out;
    p.status = a.status;
    p.rows = a.rows;
    p.rec_bytes = record_bytes(a.N, a.d, format, block);
    p.d = a.d;
    p.block = block;
    p.norm_eps = a.norm_eps;
    p.flags = a.flags;
    p.wait_polls = wait_polls;
    const CodebookParam cb = codebook_param(format);
    for (int i = 0; i < 16; ++i) p.cb[i] = cb.value[i];
    const int smem = static_cast<int>(qdecode_smem_bytes(a.N, a.d, p.rec_bytes));
    int rc = ensure_smem_opt_in(reinterpret_cast<const void *>(v.fn), smem);
    if (rc != MOLE_OK) return rc;
    void *args[1] = {&p};
    // The first of a step's layers starts on an empty machine while its blocks fill part of it only: with the launches of step after
    // step set up under one another, the blocks of a layer end up unevenly over the SMs, and stay so (8 layers of the 410M shape,
    // 256 tokens, 40 against 51 us; 12 of the 160M shape, 300 tokens, 51 against 62).  Not where an SM holds one or two blocks, or
    // so many that a few more do not matter: there the 2 us of launch count for more.
    bool alone = false;
    int sms = 0, resident = 0;
    if (a.first && !(a.flags & MOLE_FLAG_CHAIN)) {
        rc = sm_count(&sms);
        if (rc == MOLE_OK) rc = blocks_per_sm(reinterpret_cast<const void *>(v.fn), a.d / 4, smem, &resident);
        if (rc != MOLE_OK) return rc;
        alone = resident >= 3 && resident <= 8 && a.M * 2 > sms && a.M <= static_cast<long long>(resident - 1) * sms;
    }
    return launch_pdl(reinterpret_cast<const void *>(v.fn), static_cast<unsigned>(a.M), static_cast<unsigned>(a.d / 4), smem, a.stream, args,
                      (a.flags & MOLE_FLAG_CHAIN) != 0, alone);
}

// Whether a fused step over quantised tables exists for a shape (the router matrix goes through registers) and is ahead of L
// chained layers: while its tokens keep an SM to about sixteen compute warps.  12 layers, us fused against chained: 410M shape NF4
// 21.1 / 34.6 at 64 tokens, 30.7 / 67.3 at 256, even at 600; 160M NF3 34.9 / 67.3 at 256, 67.4 / 60.9 at 400; N = 16, d = 384
// 22.3 / 37.6 at 300; N = 32, d = 384 43.6 / 72.7 at 300, 111.6 / 95.9 at 1 000.
bool quant_step_preferred(long long M, int N, int d, int format, int block, int sms)
{
    if (!quant_layer_shape_ok(N, d, format, block) || d / 4 > qstep_max_threads(N)) return false;
    return M * d <= 2048LL * sms;
}

QuantVariant quant_variant(long long M, int L, int N, int d, int format, int block, bool norm, int sms)
{
    const int bits = format_bits(format);
    const long long rb = record_bytes(N, d, format, block);
    if (L > 1 && quant_step_preferred(M, N, d, format, block, sms))
        return QuantVariant{pick_qstep(N, bits, norm).name, d / 4 + 32, static_cast<int>(qstep_smem(d, rb, qstep_stages(d, rb)).total)};
    return QuantVariant{pick_qdecode(N, bits, norm).name, d / 4, static_cast<int>(qdecode_smem_bytes(N, d, rb))};
}

int launch_quant_step(const StepLaunch &a, int format, int block, uint32_t wait_polls)
{
    if (a.M == 0) return MOLE_OK;
    if (a.M * a.L > 0x3fffffffLL) return MOLE_ERR_TOO_LARGE;
    const QStepKernel fn = pick_qstep(a.N, format_bits(format), a.norm_weight != nullptr).fn;
    if (!fn || a.d / 4 > qstep_max_threads(a.N)) return MOLE_ERR_UNSUPPORTED_SHAPE;
    QStepParams p;
    p.hidden = a.hidden;
    p.row_index = a.row_index;
    p.lut = a.lut;
    p.w_router = a.w_router;
    p.norm_weight = a.norm_weight;
    p.out = a.out;
    p.status = a.status;
    p.rows = a.rows;
    p.rec_bytes = record_bytes(a.N, a.d, format, block);
    p.lut_stride = a.lut_stride;
    p.wr_stride = a.wr_stride;
    p.norm_stride = a.norm_stride;
    p.M = a.M;
    p.d = a.d;
    p.block = block;
    p.L = a.L;
    p.norm_eps = a.norm_eps;
    p.flags = a.flags;
    p.wait_polls = wait_polls;
    const CodebookParam cb = codebook_param(format);
    for (int i = 0; i < 16; ++i) p.cb[i] = cb.value[i];
    p.stages = qstep_stages(a.d, p.rec_bytes);
    const int smem = static_cast<int>(qstep_smem(a.d, p.rec_bytes, p.stages).total), threads = a.d / 4 + 32;
    int rc = ensure_smem_opt_in(reinterpret_cast<const void *>(fn), smem);
    if (rc != MOLE_OK) return rc;
    int sms = 0, per_sm = 0;
    rc = sm_count(&sms);
    if (rc != MOLE_OK) return rc;
    rc = blocks_per_sm(reinterpret_cast<const void *>(fn), threads, smem, &per_sm);
    if (rc != MOLE_OK) return rc;
    const long long resident = static_cast<long long>(per_sm) * sms;
    void *args[1] = {&p};
    return launch_pdl(reinterpret_cast<const void *>(fn), static_cast<unsigned>(a.M < resident ? a.M : resident), static_cast<unsigned>(threads), smem, a.stream, args,
                      (a.flags & MOLE_FLAG_CHAIN) != 0);
}

}  // namespace mole

using namespace mole;

extern "C" {

int mole_nf_codebook(int format, float *values)
{
    if (!values || (format != MOLE_LUT_NF4 && format != MOLE_LUT_NF3)) return MOLE_ERR_INVALID_ARG;
    const int n = 1 << format_bits(format);
    const float *src = format == MOLE_LUT_NF4 ? codebooks().nf4 : codebooks().nf3;
    for (int i = 0; i < n; ++i) values[i] = src[i];
    return MOLE_OK;
}

int mole_quant_record_bytes(int N, int d, int format, int block, int64_t *bytes)
{
    if (!bytes) return MOLE_ERR_INVALID_ARG;
    int rc = check_format(N, d, format, block);
    if (rc != MOLE_OK) return rc;
    *bytes = record_bytes(N, d, format, block);
    return MOLE_OK;
}

int mole_quantize_lut(const void *lut, void *packed, int64_t V, int N, int d, int format, int block, void *stream)
{
    int rc = check_format(N, d, format, block);
    if (rc != MOLE_OK) return rc;
    if (V < 0) return MOLE_ERR_INVALID_ARG;
    if (V == 0) return MOLE_OK;
    if (V > 0x7fffffffLL) return MOLE_ERR_TOO_LARGE;
    if (!lut || !packed || !aligned16(lut) || !aligned16(packed)) return MOLE_ERR_INVALID_ARG;
    const long long rb = record_bytes(N, d, format, block);
    const int smem = N * (d / block) * 4;
    if (smem > 48 * 1024) return MOLE_ERR_UNSUPPORTED_SHAPE;
    const CodebookParam cb = codebook_param(format);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const long long total = V * N * (d / block);
    if (block <= 2048 && total <= 0x7fffffffLL) {
        QuantGrid q;
        int cpl = 1;
        quant_group(block / 16, &q.group_log2, &cpl);
        q.rec_bytes = rb;
        q.total = static_cast<uint32_t>(total);
        q.per_id = static_cast<uint32_t>(N * (d / block));
        q.low_bytes = static_cast<uint32_t>(N) * (d / 4);
        q.code_bytes = format == MOLE_LUT_NF4 ? static_cast<uint32_t>(N) * (d / 2) : q.low_bytes + static_cast<uint32_t>(N) * (d / 8);
        q.block = block;
        q.wide_loads = (reinterpret_cast<uintptr_t>(lut) & 31u) == 0 ? 1 : 0;
        const long long per_cta = kQuantTileThreads >> q.group_log2;
        const QuantizeKernel fn = format == MOLE_LUT_NF4 ? pick_quantize<4>(cpl) : pick_quantize<3>(cpl);
        fn<<<static_cast<unsigned>((total + per_cta - 1) / per_cta), kQuantTileThreads, 0, st>>>(static_cast<const unsigned char *>(lut),
                                                                                           static_cast<unsigned char *>(packed), q, cb);
    } else if (format == MOLE_LUT_NF4) {
        mole_quantize_wide_kernel<4><<<static_cast<unsigned>(V), kQuantThreads, smem, st>>>(static_cast<const uint4 *>(lut), static_cast<unsigned char *>(packed), V, N, d, block, rb, cb);
    } else {
        mole_quantize_wide_kernel<3><<<static_cast<unsigned>(V), kQuantThreads, smem, st>>>(static_cast<const uint4 *>(lut), static_cast<unsigned char *>(packed), V, N, d, block, rb, cb);
    }
    MOLE_CUDA_TRY(cudaGetLastError());
    return MOLE_OK;
}

}  // extern "C"
