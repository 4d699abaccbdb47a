// The tensor-core form of the fused L-layer step for sm_100a (Eq. 8 of arXiv 2503.15798 applied layer after layer): one launch,
// bf16, N of 8, 16 or 32 experts, d a multiple of 128, a token per block or per cluster of blocks.
//
// What bounds a step.  One token's layer is a dependent chain -- router product, a sum over the block, a softmax, a weighted sum --
// and with one token per SM each link costs its latency plus its instructions.  On CUDA cores the weighted sum alone is three
// instructions per two elements (two unpacks and half a packed fma each).  Both products are with a small matrix, so both run on
// mma.m16n8k16 here:
//   - Router: A = W_r^T (16 experts x 16 columns per step), B = the hidden state: bf16 products, fp32 sums.
//   - Weighted sum: A = rows^T (16 columns x 16 experts), B = the softmax numerators.  A numerator is an fp32 number and is
//     never rounded: its three bf16 parts of 8 bits each are columns of the product (GateColumns).  An mma takes 8.2 cycles of a
//     quarter of an SM (measured), so that a product per part was the longest link of the chain: 16 layers of the 1B shape, 64 tokens
//     40.8 -> 36.5 us, 12 of 16 x 2048 16.1 -> 14.8, of 32 x 1024 with the norm 27.0 -> 23.9.
// Split.  Warp w owns the 128 columns 128w .. of everything: of the hidden state, of every row, of the output, and those
// columns are also its share of the router product.  So what a layer's router needs from the layer before is what the same
// warp has just computed, and warps exchange nothing but N partial logits per token: one meeting per layer.  (RMSNorm in front
// of the router adds one for the sum of squares.)  Where a token's rows exceed 32 KB a cluster of CS blocks shares the token;
// the partial logits then travel through distributed shared memory (st.async) and the meeting is an mbarrier.
// Data.  One producer warp streams router matrices and rows, whole boxes by tensor copy with the 128-byte swizzle, so that
// ldmatrix reads either without bank conflicts; a warp loads the next layer's router fragments and its rows while it waits for
// the logits of the others.
// Measured, ring kernel / here, us per step: 16 layers of the 1B shape, 64 tokens 53.2 / 36.5 (up to one block per SM: mole_slice.cuh); 10
// layers of 8 x 1024, 250 tokens 19.1 / 15.4; 12 layers with the norm, 64 tokens, of 16 x 384 30.2 / 14.8, of 16 x 2048 - / 20.4.
// The norm: a lane adds up one slice and forms one root, and the scales of the layer after stay as they were loaded until they are
// used (widened at once they were waited for at once, 300 cycles of every layer): 1B shape, 64 tokens 55.9 -> 45.7, of 16 x 2048 24.0 -> 20.4,
// of 8 x 2048 23.2 -> 21.1.
// The order of every sum is fixed by N and d: a token gets the same bits in any batch.
#pragma once

#include <cuda.h>

#include "mole_cdecode.cuh"

namespace mole {

constexpr int kMmaCols = 128;      // columns of a warp
constexpr int kMmaMaxSlots = 8;
constexpr int kMmaMaxSlices = 16;  // of a token: d <= 2048

struct MmaParams {
    const void *hidden, *row_index, *norm_weight;
    void *out;
    uint32_t *status;
    long long norm_stride;  // bytes between the scale vectors of consecutive layers
    long long rows;
    int d, L;
    int w_slots, r_slots;   // router matrices and rows of the token in flight
    float norm_eps, inv_d;
    uint32_t flags, wait_polls;
};

// Shared memory of a block: router matrices, rows, hidden slices, normalised slices, partial logits of the whole token (two
// sets), sums of squares (two sets), failure flags, barriers.
struct MmaSmem {
    uint32_t matrix;  // bytes of this block's part of a router matrix = of a token's rows
    uint32_t off_r, off_hid, off_norm, off_partial, off_ssq, off_dead, off_bars, total;
};
__host__ __device__ inline MmaSmem mma_smem(int N, int d, int cs, int w_slots, int r_slots, int norm)
{
    MmaSmem m;
    const int dl = d / cs, slices = d / kMmaCols;
    m.matrix = static_cast<uint32_t>(N) * dl * 2;
    m.off_r = static_cast<uint32_t>(w_slots) * m.matrix;
    m.off_hid = m.off_r + static_cast<uint32_t>(r_slots) * m.matrix;
    m.off_norm = m.off_hid + static_cast<uint32_t>(dl * 2);
    m.off_partial = m.off_norm + (norm ? static_cast<uint32_t>(dl * 2) : 0u);
    m.off_ssq = (m.off_partial + static_cast<uint32_t>(2 * slices * N * 4) + 15u) & ~15u;
    m.off_dead = m.off_ssq + (norm ? static_cast<uint32_t>(2 * slices * 16) : 0u);
    m.off_bars = (m.off_dead + 3 * 4 + 7u) & ~7u;
    m.total = m.off_bars + (4 * kMmaMaxSlots + 4) * 8;
    return m;
}

#ifdef __CUDACC__

__device__ __forceinline__ void tensor_load_3d(uint32_t smem_dst, const CUtensorMap *map, int c0, int c1, int c2, uint64_t *bar)
{
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                 ::"r"(smem_dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void tensor_load_5d(uint32_t smem_dst, const CUtensorMap *map, int c0, int c1, int c2, int c3, int c4, uint64_t *bar)
{
    asm volatile("cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
                 ::"r"(smem_dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void sts16(uint32_t a, unsigned short v) { asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"(v) : "memory"); }
__device__ __forceinline__ void stsf(uint32_t a, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory"); }
__device__ __forceinline__ float ldsf(uint32_t a) { return __uint_as_float(lds32(a)); }

// This warp's 128 columns of the router matrix as A fragments (experts x columns).  A matrix [columns][N] lies in rows of 128
// bytes -- 64 / N columns each -- whose 16-byte pieces are swizzled by the row number.
template <int N>
struct RouterA {
    static constexpr int ET = N == 32 ? 2 : 1;  // tiles of 16 experts
    uint32_t a[8][ET][N == 8 ? 2 : 4];          // N = 8: rows 8 .. 15 of A are zero
    uint32_t off;                               // this lane's first address inside the slice
    __device__ __forceinline__ void init(int lane)
    {
        const int i = lane & 7, m = lane >> 3;
        if constexpr (N == 8) off = static_cast<uint32_t>(m * 128 + ((i ^ m) << 4));                                               // column 8 m + i
        else if constexpr (N == 16) off = static_cast<uint32_t>((2 * (m >> 1) + (i >> 2)) * 128 + ((((i & 3) * 2 + (m & 1)) ^ (2 * (m >> 1) + (i >> 2))) << 4));
        else off = static_cast<uint32_t>((4 * (m >> 1) + (i >> 1)) * 128 + ((((i & 1) * 4 + (m & 1)) ^ (4 * (m >> 1) + (i >> 1))) << 4));
    }
    __device__ __forceinline__ void load(uint32_t slice)
    {
        if constexpr (N == 8) {
#pragma unroll
            for (int s = 0; s < 8; s += 2) {  // two steps of 16 columns per load
                uint32_t r[4];
                ldsm_x4_trans(r, (slice + off + static_cast<uint32_t>(s) * 256u) ^ ((s & 2) ? 64u : 0u));
                a[s][0][0] = r[0], a[s][0][1] = r[1], a[s + 1][0][0] = r[2], a[s + 1][0][1] = r[3];
            }
        } else if constexpr (N == 16) {
#pragma unroll
            for (int s = 0; s < 8; ++s) ldsm_x4_trans(a[s][0], (slice + off + static_cast<uint32_t>(s) * 512u) ^ ((s & 1) ? 64u : 0u));
        } else {
#pragma unroll
            for (int s = 0; s < 8; ++s)
#pragma unroll
                for (int e = 0; e < 2; ++e) ldsm_x4_trans(a[s][e], (slice + off + static_cast<uint32_t>(s) * 1024u) ^ (e ? 32u : 0u));
        }
    }
    // z[e]: fragment of expert tile e over the slice; steps in four chains.  h: this lane's ldmatrix address in the hidden slice(s)
    __device__ __forceinline__ void product(uint32_t h, float (&z)[ET][4]) const
    {
        uint32_t b[4][4];
#pragma unroll
        for (int s = 0; s < 4; ++s) ldsm_x4(b[s], h + 64u * s);
        float c[ET][4][4];
#pragma unroll
        for (int e = 0; e < ET; ++e)
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int i = 0; i < 4; ++i) c[e][k][i] = 0.f;
#pragma unroll
        for (int s = 0; s < 8; ++s)
#pragma unroll
            for (int e = 0; e < ET; ++e) {
                const uint32_t b0 = b[s >> 1][2 * (s & 1)], b1 = b[s >> 1][2 * (s & 1) + 1];
                if constexpr (N == 8) mma16(c[e][s & 3], a[s][0][0], 0u, a[s][0][1], 0u, b0, b1);
                else mma16(c[e][s & 3], a[s][e][0], a[s][e][1], a[s][e][2], a[s][e][3], b0, b1);
            }
#pragma unroll
        for (int e = 0; e < ET; ++e)
#pragma unroll
            for (int i = 0; i < 4; ++i) z[e][i] = (c[e][0][i] + c[e][1][i]) + (c[e][2][i] + c[e][3][i]);
    }
};

// A token's softmax numerators as B fragments (experts x 8 columns).  A numerator is an fp32 number >= 0 and is not rounded: it is
// hi + mid + lo, three bf16 parts of 8 bits each.  Columns 0 - 2 of the product are the parts, columns 4 - 6 the same again: one
// product per tile and step, of which a lane with even q has the sums of hi and mid and its neighbour that of lo (RowsA).
// A mid or lo of zero beside a hi that is not becomes 2^-126, the smallest normal number (and so is column 3): zero times an infinite
// table entry would be NaN where the number times it is infinite, and the sums of finite entries, whose largest numerator is
// 2^-87 at least, do not see it.
template <int N>
struct GateColumns {
    static constexpr int KS = N == 32 ? 2 : 1;  // steps of 16 experts
    static constexpr int W = N == 8 ? 1 : 2;    // words per step
    uint32_t b[KS][W];
    float esum;  // of this lane's numerators; summed over q: of all
    // e: lane first + j holds the numerator of expert j
    __device__ __forceinline__ void from_lanes(float e, int lane, int first)
    {
        const int q = lane & 3, part = (lane >> 2) & 3;
        const bool p0 = part == 0, p1 = part == 1, p2 = part == 2;
        float v[2 * W * KS];
#pragma unroll
        for (int i = 0; i < 2 * W * KS; ++i) v[i] = __shfl_sync(0xffffffffu, e, first + 8 * (i >> 1) + 2 * q + (i & 1));
        esum = 0.f;
#pragma unroll
        for (int w = 0; w < W * KS; ++w) {
            float x[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float a = v[2 * w + i], ar = a - __uint_as_float(__float_as_uint(a) & 0xffff0000u);
                const float al = ar - __uint_as_float(__float_as_uint(ar) & 0xffff0000u);
                x[i] = p0 ? a : (p1 ? ar : (p2 ? al : 0.f));
            }
            const uint32_t hi = __byte_perm(__float_as_uint(v[2 * w]), __float_as_uint(v[2 * w + 1]), 0x7632);
            b[w / W][w % W] = __vmaxu2(__byte_perm(__float_as_uint(x[0]), __float_as_uint(x[1]), 0x7632), __vminu2(hi, 0x00800080u));
            esum += v[2 * w] + v[2 * w + 1];
        }
    }
    __device__ __forceinline__ float sum() const
    {
        const float s = esum + __shfl_xor_sync(0xffffffffu, esum, 1);
        return s + __shfl_xor_sync(0xffffffffu, s, 2);
    }
};

// This warp's 128 columns of a token's rows as A fragments (columns x experts): eight tiles of 16 columns.  The rows lie as
// [64-column chunk][expert][128 bytes], 16-byte pieces swizzled by the expert.
template <int N>
struct RowsA {
    static constexpr int KS = GateColumns<N>::KS, W = GateColumns<N>::W;
    uint32_t a[8][KS][2 * W];
    static __device__ __forceinline__ uint32_t lane_offset(int lane)
    {
        const int i = lane & 7, m = lane >> 3;
        if constexpr (N == 8) return static_cast<uint32_t>(i * 128 + ((i ^ m) << 4));  // piece m of four: two tiles per load
        else return static_cast<uint32_t>((i + 8 * (m >> 1)) * 128 + ((i ^ (m & 1)) << 4));
    }
    __device__ __forceinline__ void load(uint32_t addr)  // slot + this warp's chunks + lane offset
    {
        if constexpr (N == 8) {
#pragma unroll
            for (int t = 0; t < 8; t += 2) {
                uint32_t r[4];
                ldsm_x4_trans(r, (addr + static_cast<uint32_t>(t >> 2) * (N * 128u)) ^ ((t & 2) ? 64u : 0u));
                a[t][0][0] = r[0], a[t][0][1] = r[1], a[t + 1][0][0] = r[2], a[t + 1][0][1] = r[3];
            }
        } else {
#pragma unroll
            for (int t = 0; t < 8; ++t)
#pragma unroll
                for (int k = 0; k < KS; ++k)
                    ldsm_x4_trans(a[t][k], (addr + static_cast<uint32_t>(t >> 2) * (N * 128u) + static_cast<uint32_t>(k) * 2048u) ^ (static_cast<uint32_t>(t & 3) << 5));
        }
    }
    // v[i]: the sums of this lane's four columns: 16 q + r, 16 q + 8 + r, 64 + 16 q + r, 64 + 16 q + 8 + r  (lane = 4 r + q); `under` is
    // done while the products are on their way
    template <typename F>
    __device__ __forceinline__ void product(const GateColumns<N> &g, int lane, float (&v)[4], F &&under) const
    {
        float c[8][4];
#pragma unroll
        for (int t = 0; t < 8; ++t)
#pragma unroll
            for (int i = 0; i < 4; ++i) c[t][i] = 0.f;
#pragma unroll
        for (int k = 0; k < KS; ++k)
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                if constexpr (N == 8) mma8(c[t], a[t][k][0], a[t][k][1], g.b[k][0]);
                else mma16(c[t], a[t][k][0], a[t][k][1], a[t][k][2], a[t][k][3], g.b[k][0], g.b[k][1]);
            }
        under();
        const bool q0 = (lane & 1) != 0, q1 = (lane & 2) != 0;  // lane q takes tiles q and 4 + q, the rest of their sums from its neighbour
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int base = (i >> 1) * 4, w = (i & 1) * 2;
            float s[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) s[t] = c[base + t][w] + c[base + t][w + 1];
            const float even = q1 ? s[2] : s[0], odd = q1 ? s[3] : s[1];
            v[i] = (q0 ? odd : even) + __shfl_xor_sync(0xffffffffu, q0 ? even : odd, 1);
        }
    }
};

// 1 / sqrt(x) to within an ulp for x >= 0, infinities included: the hardware's reciprocal root and a Newton step whose residual
// 1 - x r^2 is taken without a rounding of x r (two roundings of the correctly rounded root and division are no closer).
__device__ __forceinline__ float rsqrt_refined(float x)
{
    const float r = rsqrtf(x), s = x * r;
    const float e = fmaf(-fmaf(x, r, -s), r, fmaf(-s, r, 1.0f));
    return x > 0.f && x < INFINITY ? fmaf(0.5f * r, e, r) : r;
}

// Softmax numerator of a logit; `group`: lanes (a power of two) that hold one token's logits.  The maximum is subtracted only
// where a token has a logit beyond +-60 (exp and the parts of its result then leave the normal range): any shift gives the same gates.
__device__ __forceinline__ float softmax_part(float z, int group)
{
    float shift = 0.f;
    if (__any_sync(0xffffffffu, !(fabsf(z) < 60.f))) {
        float zm = z;
        int big = !(fabsf(z) < 60.f) ? 1 : 0;
        for (int o = group / 2; o >= 1; o >>= 1) {
            zm = fmaxf(zm, __shfl_xor_sync(0xffffffffu, zm, o));
            big |= __shfl_xor_sync(0xffffffffu, big, o);
        }
        if (big) shift = zm;
    }
    return expf(z - shift);
}

// N: experts.  NORM: the router reads RMSNorm(hidden).  CS: blocks per token.
// Registers: for two blocks per SM (at most 96; N = 16 without pairs spills 16 bytes, with the norm 32), but where that spills on the
// critical path or two large blocks rarely meet: N = 32 (168), and N = 16 in pairs (119, with the norm 134; 12 layers of 16 x 2048 with the norm, 64 tokens 33.5 -> 24.0 us, of 16 x 1280 29.5 -> 21.5).
// Launch: d / CS / 4 + 32 threads, mma_smem(..).total bytes, CS blocks per token.
template <int N, int NORM, int CS>
__global__ void __cluster_dims__(CS, 1, 1) __launch_bounds__(8 * 32 + 32, N == 32 || (N == 16 && CS == 2) ? 1 : 2)
    mole_mma_kernel(const __grid_constant__ CUtensorMap w_map, const __grid_constant__ CUtensorMap r_map, const MmaParams p)
{
    constexpr int ET = RouterA<N>::ET;
    extern __shared__ __align__(1024) unsigned char smem_1k[];
    unsigned char *const smem = smem_1k;

    pdl_enter(p.flags);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = static_cast<int>(blockDim.x >> 5) - 1;
    const int d = p.d, L = p.L, WS = p.w_slots, RS = p.r_slots, slices = nw * CS;
    const uint32_t rank = CS > 1 ? cluster_ctarank() : 0u;
    const MmaSmem m = mma_smem(N, d, CS, WS, RS, NORM);
    const uint32_t base = smem_u32(smem);
    volatile int *dead = reinterpret_cast<volatile int *>(smem + m.off_dead);  // somebody gave up waiting
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + m.off_bars);
    uint64_t *wfull = bars, *wempty = bars + kMmaMaxSlots, *rfull = bars + 2 * kMmaMaxSlots, *rempty = bars + 3 * kMmaMaxSlots;
    uint64_t *xbar = bars + 4 * kMmaMaxSlots, *sbar = xbar + 2;  // the cluster's exchanges: logits, sums of squares
    const size_t t = blockIdx.x / CS;                            // this block's token

    if (tid == 0) {
        for (int s = 0; s < WS; ++s) {
            mbar_init(wfull + s, 1);
            mbar_init(wempty + s, nw);
        }
        for (int s = 0; s < RS; ++s) {
            mbar_init(rfull + s, 1);
            mbar_init(rempty + s, nw);
        }
        for (int s = 0; s < 4; ++s) mbar_init(xbar + s, 1);
        dead[0] = 0;
        dead[2] = 0;  // raised by nobody: the drain waits run their (short) course
        mbar_init_fence();
    }
    __syncthreads();
    if constexpr (CS > 1) cluster_arrive();  // waited for before the first push

    if (warp == nw) {
        // ================= producer warp: copies in the order they are consumed -- the first router matrix, then per layer
        // the token's rows and the router matrix of the layer after =================
        int ws = 0, rs = 0, issued_w = 0, issued_r = 0;
        uint32_t wph = 1, rph = 1;  // parity of the `empty` phase that frees the slot
        bool ok = true;
        const int w_rows = nw * (2 * N);  // 128-byte rows of this block's part of a router matrix, at most 256
        auto wait_slot = [&](uint64_t *bar, uint32_t parity) {
            int got = 1;
            if (lane == 0) {
                got = wait_or_give_up(bar, parity, dead, p.wait_polls, true);
                if (!got) report_timeout(dead, p.status);
            }
            ok = __shfl_sync(0xffffffffu, got, 0) != 0;
        };
        auto issue_router = [&]() {
            if (issued_w >= L) return;
            if (issued_w >= WS) wait_slot(wempty + ws, wph);
            if (!ok) return;
            if (lane == 0) {
                mbar_expect_tx(wfull + ws, m.matrix);
                tensor_load_3d(base + static_cast<uint32_t>(ws) * m.matrix, &w_map, 0, static_cast<int>(rank) * w_rows, issued_w, wfull + ws);
            }
            ++issued_w;
            if (++ws == WS) ws = 0, wph ^= 1u;
        };
        issue_router();
        const int id = __ldg(static_cast<const int *>(p.row_index) + t);
        const bool valid = id >= 0 && id < p.rows;
        if (!valid && lane == 0 && rank == 0 && p.status) atomicOr(p.status, MOLE_STATUS_BAD_ID);
#pragma unroll 1
        for (int l = 0; l < L && ok; ++l) {
            if (issued_r >= RS) wait_slot(rempty + rs, rph);
            if (!ok) break;
            if (lane == 0) {
                if (valid) {
                    mbar_expect_tx(rfull + rs, m.matrix);
                    tensor_load_5d(base + m.off_r + static_cast<uint32_t>(rs) * m.matrix, &r_map, 0, 0, static_cast<int>(rank) * nw * 2, id, l, rfull + rs);
                } else {
                    mbar_arrive(rfull + rs);  // nothing to copy: the routed term is dropped
                }
            }
            ++issued_r;
            if (++rs == RS) rs = 0, rph ^= 1u;
            issue_router();
        }
        if (*dead) {
            drain_ring(wfull, WS, issued_w);
            drain_ring(rfull, RS, issued_r);
        }
        __syncwarp();
        if constexpr (CS > 1) cluster_wait();
    } else {
        // ================= compute warps ======================================================================================
        const int nc = nw * 32;
        const int slice = static_cast<int>(rank) * nw + warp;  // of the whole token
        const int r8 = lane >> 2, q = lane & 3;
        const uint32_t hid = base + m.off_hid + static_cast<uint32_t>(warp) * (kMmaCols * 2);
        const uint32_t router_in = (NORM ? base + m.off_norm + static_cast<uint32_t>(warp) * (kMmaCols * 2) : hid);
        const uint32_t own_off = static_cast<uint32_t>(2 * (16 * q + r8));  // this lane's columns: + 0, 16, 128, 144 bytes
        auto col = [](int i) -> uint32_t { return static_cast<uint32_t>((i >> 1) * 128 + (i & 1) * 16); };
        const uint32_t part_set = static_cast<uint32_t>(slices * N * 4);
        const uint32_t w_off = static_cast<uint32_t>(warp) * (256u * N);
        const uint32_t r_off = m.off_r + static_cast<uint32_t>(warp) * (256u * N) + RowsA<N>::lane_offset(lane);
        const size_t slice_bytes = static_cast<size_t>(slice) * (kMmaCols * 2);
        bool alive = true;  // false after a wait ran out: no more waiting, whatever is there is computed on (the status says so)
        auto acquire = [&](uint64_t *bar, uint32_t parity) {
            if (alive && mbar_try_wait(bar, parity)) return;
            alive = acquire_slow(bar, parity, dead, alive, true, p.status, lane, p.wait_polls);
        };
        auto acquire_cluster = [&](uint64_t *bar, uint32_t parity) {
            for (uint32_t i = 0; alive; ++i) {
                if (mbar_try_wait_cluster(bar, parity)) return;
                if (i >= p.wait_polls) {
                    if (lane == 0) report_timeout(dead, p.status);
                    alive = false;
                }
                if (i > 64) __nanosleep(32);
                if ((i & 127u) == 127u && *dead) alive = false;
            }
        };
        int ws = 0, rs = 0;
        uint32_t wph = 0, rph = 0;
        RouterA<N> wf;
        wf.init(lane);
        auto load_router = [&]() {
            acquire(wfull + ws, wph);
            wf.load(base + static_cast<uint32_t>(ws) * m.matrix + w_off);
        };
        load_router();
        if constexpr (CS > 1) cluster_wait();
        const int id = __ldg(static_cast<const int *>(p.row_index) + t);
        const bool valid = id >= 0 && id < p.rows;

        pdl_wait();

        const size_t token_bytes = t * d * 2 + slice_bytes + (lane & 15) * 16;  // lanes 0-15: this warp's columns, 16 bytes each
        if (lane < 16) cp_async16(hid + lane * 16, static_cast<const unsigned char *>(p.hidden) + token_bytes);
        cp_async_commit();
        const unsigned char *norm_g = static_cast<const unsigned char *>(p.norm_weight) + slice_bytes + own_off;
        unsigned short wgt_next[4] = {0, 0, 0, 0};  // as loaded: widened here they would be waited for here
        auto load_norm = [&](int l) {
#pragma unroll
            for (int i = 0; i < 4; ++i) wgt_next[i] = __ldg(reinterpret_cast<const unsigned short *>(norm_g + static_cast<size_t>(l) * p.norm_stride + col(i)));
        };
        if constexpr (NORM) load_norm(0);

        uint32_t buf = 0, xph = 0;  // exchange buffer, its barrier's parity
        cp_async_wait_all();
        __syncwarp();
        float h[4];  // this lane's columns of the running hidden state
#pragma unroll
        for (int i = 0; i < 4; ++i) h[i] = bf16_bits_to_float(lds16(hid + own_off + col(i)));
#pragma unroll 1
        for (int l = 0; l < L; ++l) {
            const bool last = l == L - 1;
            if (CS > 1 && tid == 0) {
                mbar_expect_tx(xbar + buf, part_set);
                if (NORM) mbar_expect_tx(sbar + buf, static_cast<uint32_t>(slices * 16));
            }
            if constexpr (NORM) {
                // y = (x / sqrt(mean(x^2) + eps)) * w, rounded once to bf16: what the router reads
                const uint32_t sq = base + m.off_ssq + buf * static_cast<uint32_t>(slices * 16);
                float ss = fmaf(h[1], h[1], h[0] * h[0]) + fmaf(h[3], h[3], h[2] * h[2]);
#pragma unroll
                for (int o = 16; o >= 4; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
                if (lane < 4 * CS) {  // (the sums are the same in all lanes with the same last two bits)
                    const uint32_t at = sq + static_cast<uint32_t>(slice * 4 + (lane & 3)) * 4u, to = static_cast<uint32_t>(lane) >> 2;
                    if constexpr (CS == 1) stsf(at, ss);
                    else cluster_push_f32(cluster_map(at, to), ss, cluster_map(smem_u32(sbar + buf), to));
                }
                if constexpr (CS == 1) named_bar_sync(3, nc);
                else acquire_cluster(sbar + buf, xph);
                // lane l adds up slice l % 16, then they add up each other's: one load and one root per lane
                const int from = lane & 15;
                const uint4 part = lds128(sq + static_cast<uint32_t>(from < slices ? from : 0) * 16u);
                float total = (__uint_as_float(part.x) + __uint_as_float(part.y)) + (__uint_as_float(part.z) + __uint_as_float(part.w));
                if (from >= slices) total = 0.f;
#pragma unroll
                for (int o = 8; o >= 1; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
                // total / d, correctly rounded (an infinite total would make the correction NaN)
                float mean = total * p.inv_d;
                mean = total < INFINITY ? fmaf(fmaf(-mean, static_cast<float>(d), total), p.inv_d, mean) : total;
                const float rinv = rsqrt_refined(mean + p.norm_eps);
#pragma unroll
                for (int i = 0; i < 4; ++i) sts16(router_in + own_off + col(i), float_to_bf16_bits((h[i] * rinv) * bf16_bits_to_float(wgt_next[i])));
                if (!last) load_norm(l + 1);
                __syncwarp();
            }

            // ---- router: this warp's partial logits: lane 4 r holds experts r, r + 8 ----
            float z[ET][4];
            wf.product(router_in + static_cast<uint32_t>(lane >> 3) * 16u, z);
            const uint32_t part = base + m.off_partial + buf * part_set;
            if (q == 0) {
#pragma unroll
                for (int e = 0; e < ET; ++e)
#pragma unroll
                    for (int i = 0; i < (N == 8 ? 1 : 2); ++i) {
                        const uint32_t at = part + static_cast<uint32_t>(slice * N + 16 * e + r8 + 8 * i) * 4u;
                        if constexpr (CS == 1) stsf(at, z[e][2 * i]);
                        else
#pragma unroll
                            for (int c = 0; c < CS; ++c) cluster_push_f32(cluster_map(at, c), z[e][2 * i], cluster_map(smem_u32(xbar + buf), c));
                    }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(wempty + ws);  // the matrix has been multiplied: its slot goes back
            if (++ws == WS) ws = 0, wph ^= 1u;
            if constexpr (CS == 1) named_bar_arrive(1, 2 * nc);
            // under the others' products: this token's rows, the next router matrix
            acquire(rfull + rs, rph);
            RowsA<N> rows;
            rows.load(base + static_cast<uint32_t>(rs) * m.matrix + r_off);
            if (!last) load_router();
            if constexpr (CS == 1) named_bar_sync(1, 2 * nc);
            else acquire_cluster(xbar + buf, xph);

            // ---- softmax numerators (Eq. 4), by every warp for itself: even slices and odd slices, then the two ----
            float e;
            {
                const uint32_t z_in = part + static_cast<uint32_t>(lane & (N - 1)) * 4u;
                float v[kMmaMaxSlices], ze = 0.f, zo = 0.f;
#pragma unroll
                for (int w = 0; w < kMmaMaxSlices; ++w) v[w] = w < slices ? ldsf(z_in + static_cast<uint32_t>(w * N) * 4u) : 0.f;
#pragma unroll
                for (int w = 0; w < kMmaMaxSlices; w += 2) ze += v[w], zo += v[w + 1];
                e = softmax_part(ze + zo, N);
            }
            // ---- weighted sum of the rows (Eq. 8), residual, one rounding ----
            float v[4], inv;
            GateColumns<N> g;
            g.from_lanes(e, lane, 0);
            rows.product(g, lane, v, [&]() { inv = __frcp_rn(g.sum()); });
            __syncwarp();
            if (lane == 0) mbar_arrive(rempty + rs);
            if (++rs == RS) rs = 0, rph ^= 1u;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const unsigned short o = float_to_bf16_bits(valid ? fmaf(v[i], inv, h[i]) : h[i]);
                h[i] = bf16_bits_to_float(o);
                if (!NORM || last) sts16(hid + own_off + col(i), o);
            }
            __syncwarp();
            buf ^= 1u;
            if (buf == 0) xph ^= 1u;
        }
        if (lane < 16) *reinterpret_cast<uint4 *>(static_cast<unsigned char *>(p.out) + token_bytes) = lds128(hid + lane * 16);
        if (CS > 1 && !alive)  // the other blocks' pushes have not been waited for: time to land, before the blocks can exit
            for (int i = 0; i < 32; ++i) __nanosleep(1000);
    }
    if constexpr (CS > 1) {  // pushes to this block may still be on their way: nobody leaves before everybody is done
        cluster_arrive();
        cluster_wait();
    }
}

#endif  // __CUDACC__

}  // namespace mole
