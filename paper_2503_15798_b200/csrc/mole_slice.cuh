// The layer and the fused L-layer step of the two narrow widths of the paper's Table 2 (N = 16 experts, d = 768 and 1024, bf16) for
// sm_100a (slice_layer<d,T,NORM,LOOP> and slice_step<N,d,T,NORM,CS> to mole_variant), and the fused step of its widest (N = 32, d = 2048)
// while every token has four SMs to itself, the bits of mma<32,..,4>.  (Eq. 4 and Eq. 8 of arXiv 2503.15798.)
// Which widths: the paper's, each of which had a ring kernel with its sizes compiled in before, and costs a dozen instantiations.  Nothing
// here is about them: the kernels take an even number of warps (d a multiple of 256), as far as slots and registers reach.  A neighbour run
// through them, 12 fused layers of 16 x 512, us, mole_mma.cuh / here: 64 tokens 10.6 / 9.8, 140 tokens 10.7 / 8.9, 256 tokens 12.9 / 11.1, with
// the norm 15.4 / 13.9, 15.6 / 12.1, 18.5 / 14.3.
//
// What bounds them.  A token's layer is a dependent chain -- router product, a sum over the block, a softmax, a weighted sum -- and a
// decode batch has one or two tokens per SM, so a layer costs the length of the chain, and what it shares the chip's queues with: the
// shared-memory port takes a warp's requests in order, so a late load of 16 ldmatrix delays a partial logit behind it.  Here:
//   - Warp w owns the 128 columns 128w .. of everything: of the hidden state, of the rows, of the output, of the router product.
//     Warps exchange nothing but 16 partial logits per token: one block barrier per layer (and one for the norm).
//   - Both products run on mma.m16n8k16, as in mole_mma.cuh.  A numerator's three bf16 parts are columns of one product
//     (GateColumns): at 8.2 cycles an mma and quarter of an SM (measured) three products took 400 cycles of a layer, one takes 200.
//   - Four warps (beside a cluster's four: one) do nothing but copy rows and router matrices into swizzled slots (cp.async).  They take part in the layer's barrier,
//     which so is the handshake, too: no mbarrier is polled.  The other warps take an item from its slot into registers while they
//     compute the softmax and the weighted sum of the item before.
//   - Widths, warps and slots are compile-time, so the chain has no loop or bound to evaluate.
// How many blocks and tokens (slice_plan_d): a fused step of up to half a token per SM gives a token to a cluster of two blocks, which
// halves the bytes through either port (64 KB a layer and SM at d = 1024, 512 cycles in and 512 out) and pays 250 cycles for the exchange: 24
// layers of d = 1024, 64 tokens 22.2 -> 18.9 us, with the norm 29.1 -> 26.6, 12 layers of 768 11.3 -> 10.5.  Up to one token per SM a
// block has one token.  Beyond, a block has two, which share the router fragments (as columns of one product) and its bytes.
// Measured, us per step, ring kernel with the sizes compiled in / here.  Fused, 12 layers of 768: 64 tokens 14.3 / 10.5, 256 tokens
// 17.3 / 14.3, 1000 tokens 60.8 / 51.5; 24 layers of 1024: 64 tokens 27.7 / 18.9, with the norm 34.7 / 26.6; 256 tokens 37.1 / 35.2, with
// the norm 44.7 / 40.3; 1000 tokens 173 / 129.  Chained, 256 tokens: 12 of 768 35.8 / 31.4, 24 of 1024 73.6 / 72.0 (up to 148 tokens
// the host's launches are what is left: 2.2 us each).  Of a layer's 1 300 cycles at 64 tokens of d = 1024: router product 125, exchange and loads 370, logits
// and exp 200, parts of the numerators 95, weighted sum and output 300.
// The widest layer, 16 layers, 16 tokens, mole_mma.cuh / here: 25.2 / 18.2, with the norm 35.7 / 27.7.  Beyond one block per SM a second
// round of clusters is no faster than two blocks per SM there (64 tokens 43.7 against 36.5, with the norm 54.9 against 45.7).
// Tried: rows straight from L2 to registers, packed with byte permutes (no slots, half the port's bytes, but one layer of lead is too
// little for L2's latency: 256 tokens 14.5 -> 25.8 us); slots freed by a barrier of their own, half a layer earlier (14.5 -> 15.8).
// The order of every sum is that of one token and fixed by d: single layers, chained and fused steps and any batch give the same bits.
#pragma once

#include "mole_mma.cuh"

namespace mole {

// copying warps of a fused step: one per quarter of the SM; one in all beside a cluster's four warps
__host__ __device__ constexpr int slice_copy_warps(int N) { return N == 16 ? 4 : 1; }
// of a warp: its columns of a router matrix, or of a token's rows
__host__ __device__ constexpr uint32_t slice_bytes(int N) { return static_cast<uint32_t>(kMmaCols * N * 2); }

// Shared memory of a block of NW warps and T tokens with S slots: [slot][router | token rows][warp] slices, hidden and normalised
// slices [warp][token], partial logits [2][warp][token][expert], sums of squares [2][token][warp][4], a barrier and a flag.
struct SliceSmem {
    uint32_t slot, off_hid, off_norm, off_partial, off_ssq, off_bar, total;
};
__host__ __device__ constexpr SliceSmem slice_smem(int N, int nw, int tokens, int slots, int norm, int cs = 1)
{
    SliceSmem m{};
    m.slot = static_cast<uint32_t>(nw) * slice_bytes(N) * static_cast<uint32_t>(1 + tokens);
    m.off_hid = m.slot * static_cast<uint32_t>(slots);
    const uint32_t state = static_cast<uint32_t>(nw * tokens * kMmaCols * 2);
    m.off_norm = m.off_hid + state;
    m.off_partial = m.off_norm + (norm ? state : 0u);
    m.off_ssq = m.off_partial + static_cast<uint32_t>(2 * cs * nw * tokens * N * 4);
    m.off_bar = m.off_ssq + (norm ? static_cast<uint32_t>(2 * cs * nw * tokens * 16) : 0u);
    m.total = m.off_bar + 48u;
    return m;
}
// slots of a fused step: as many as fit (a block has the SM to itself)
__host__ __device__ constexpr int slice_slots(int N, int nw, int tokens, int cs = 1)
{
    int s = 4;
    while (s > 2 && slice_smem(N, nw, tokens, s, 1, cs).total > 227u * 1024u) --s;
    return s;
}

#ifdef __CUDACC__

template <int PENDING>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory"); }

// This warp's N x 128 slice of a token's rows (row: the first expert's row, at the warp's columns) into a slot: [64-column
// half][expert][128 bytes], 16-byte pieces swizzled by the expert (RowsA).
template <int N, int D>
__device__ __forceinline__ void slice_copy_rows(uint32_t slot, const unsigned char *row, int lane)
{
    const uint32_t e = static_cast<uint32_t>(lane) >> 4, piece = static_cast<uint32_t>(lane) & 15u;
    const uint32_t dst = slot + (piece >> 3) * (N * 128u) + e * 128u + (((piece & 7u) ^ e) << 4);
    const unsigned char *src = row + e * (D * 2u) + piece * 16u;
#pragma unroll
    for (uint32_t i = 0; i < N / 2; ++i) cp_async16((dst ^ ((2u * i & 6u) << 4)) + i * 256u, src + i * (D * 4u));
}
// ... its 128 x N slice of a router matrix (one piece): rows of 128 bytes, 64 / N columns each, 16-byte pieces swizzled by
// the row (RouterA)
template <int N>
__device__ __forceinline__ void slice_copy_router(uint32_t slot, const unsigned char *w, int lane)
{
    const uint32_t row = static_cast<uint32_t>(lane) >> 3, within = static_cast<uint32_t>(lane) & 7u;
    const uint32_t dst = slot + row * 128u + ((within ^ row) << 4);
    const unsigned char *src = w + lane * 16;
#pragma unroll
    for (uint32_t i = 0; i < N / 2; ++i) cp_async16((dst ^ ((i & 1u) << 6)) + i * 512u, src + i * 512u);
}

// One layer of a block's T tokens from the fragments on: what single layers and fused steps have in common.
// COUNT: threads at the layer's barrier.  CS: blocks of a cluster that share the token, each NB of its slices: the barrier is then an
// mbarrier of each block (mbar + 0, 1 by turns), at which the partial logits pushed into it are counted in, and likewise for the
// sums of squares (mbar + 2, 3).
template <int N, int D, int T, int NORM, int COUNT_, int CS = 1>
struct SliceLayer {
    static constexpr int NW = D / kMmaCols, NB = NW / CS, NC = NB * 32, COUNT = COUNT_;
    static_assert(CS == 1 || T == 1, "a cluster owns one token");
    static constexpr int kBarLogits = 1, kBarSquares = 2;
    uint32_t hid, normed, partial, ssq;  // this warp's hidden / normalised slices; the block's exchange areas
    uint32_t own_off;                    // this lane's first column of a slice, in bytes: it has columns + 0, 16, 128, 144 bytes
    uint32_t b_off;                      // this lane's ldmatrix address in a warp's slices
    int lane, warp, slice;               // warp of the block, slice of the token
    float h[T][4];                       // this lane's columns of the running hidden state
    uint64_t *mbar;
    volatile int *dead;
    uint32_t *status;
    uint32_t polls, phase;
    bool alive;                          // false after a wait ran out: nothing waits any more, the status says so

    static __device__ __forceinline__ uint32_t col(int i) { return static_cast<uint32_t>((i >> 1) * 128 + (i & 1) * 16); }

    __device__ __forceinline__ void init(uint32_t base, const SliceSmem &m)
    {
        lane = static_cast<int>(threadIdx.x) & 31, warp = static_cast<int>(threadIdx.x) >> 5;
        slice = CS == 1 ? warp : static_cast<int>(cluster_ctarank()) * NB + warp;
        phase = 0;
        alive = true;
        constexpr uint32_t state = T * kMmaCols * 2;
        hid = base + m.off_hid + static_cast<uint32_t>(warp) * state;
        normed = base + m.off_norm + static_cast<uint32_t>(warp) * state;
        partial = base + m.off_partial;
        ssq = base + m.off_ssq;
        own_off = static_cast<uint32_t>(2 * (16 * (lane & 3) + (lane >> 2)));
        // matrix lane / 8 of four: 8 columns; its row n is column n of the product: all of one token, or 0 - 3 and 4 - 7 of two
        b_off = static_cast<uint32_t>(lane >> 3) * 16u + (T == 2 ? static_cast<uint32_t>((lane & 7) >> 2) * (kMmaCols * 2u) : 0u);
    }
    __device__ __forceinline__ void wait_cluster(uint64_t *bar)
    {
        for (uint32_t i = 0; alive; ++i) {
            if (i >= polls) {
                if (lane == 0) report_timeout(dead, status);
                alive = false;
                return;
            }
            if (mbar_try_wait_cluster(bar, phase)) return;
            if (i > 64) __nanosleep(32);
            if ((i & 127u) == 127u && *dead) alive = false;
        }
    }
    // before a layer (one thread): what its exchanges will bring
    __device__ __forceinline__ void arm(uint32_t buf)
    {
        if constexpr (CS > 1) {
            if (threadIdx.x == 0 && alive) {  // (a barrier whose phase was not waited for takes no arrivals of the next)
                mbar_expect_tx(mbar + buf, NW * N * 4);
                if (NORM) mbar_expect_tx(mbar + 2 + buf, NW * 16);
            }
        }
    }
    // 16 lanes fetch a token's 128 columns (token: lane / 16 of two); out of range: nothing.  With the norm,
    // `under` is done while they are on their way
    template <typename F>
    __device__ __forceinline__ void load_hidden(const unsigned char *hidden, long long t0, long long M, F &&under)
    {
        const long long t = t0 + (T == 2 ? lane >> 4 : 0);
        auto load = [&]() { return __ldcg(reinterpret_cast<const uint4 *>(hidden + static_cast<size_t>(t) * (D * 2) + slice * 256 + (lane & 15) * 16)); };
        if constexpr (NORM) {
            const bool mine = (T == 2 || lane < 16) && t < M;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (mine) v = load();
            under();
            if (mine) sts128(hid + static_cast<uint32_t>(lane) * 16u, v);
        } else {
            if ((T == 2 || lane < 16) && t < M) sts128(hid + static_cast<uint32_t>(lane) * 16u, load());
        }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < T; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) h[j][i] = bf16_bits_to_float(static_cast<unsigned short>(lds16(hid + static_cast<uint32_t>(j) * 256u + own_off + col(i))));
    }
    __device__ __forceinline__ void store_out(unsigned char *out, long long t0, long long M)
    {
        __syncwarp();
        const long long t = t0 + (T == 2 ? lane >> 4 : 0);
        if ((T == 2 || lane < 16) && t < M)
            *reinterpret_cast<uint4 *>(out + static_cast<size_t>(t) * (D * 2) + slice * 256 + (lane & 15) * 16) = lds128(hid + static_cast<uint32_t>(lane) * 16u);
    }
    // y = (x / sqrt(mean(x^2) + eps)) * w, rounded once to bf16, into the normalised slices
    template <typename W>  // bf16 bits
    __device__ __forceinline__ void normalise(const W (&w)[4], float eps, uint32_t buf)
    {
        const uint32_t sq = ssq + buf * static_cast<uint32_t>(NW * T * 16);
#pragma unroll
        for (int j = 0; j < T; ++j) {
            float s = fmaf(h[j][1], h[j][1], h[j][0] * h[j][0]) + fmaf(h[j][3], h[j][3], h[j][2] * h[j][2]);
#pragma unroll
            for (int o = 16; o >= 4; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if constexpr (CS == 1) {
                if (lane < 4) stsf(sq + static_cast<uint32_t>((j * NW + warp) * 4 + lane) * 4u, s);
            } else {
                if (lane < 4 * CS) {  // (the sums are the same in all lanes with the same last two bits)
                    const uint32_t at = sq + static_cast<uint32_t>(slice * 4 + (lane & 3)) * 4u, to = static_cast<uint32_t>(lane) >> 2;
                    cluster_push_f32(cluster_map(at, to), s, cluster_map(smem_u32(mbar + 2 + buf), to));
                }
            }
        }
        if constexpr (CS == 1) named_bar_sync(kBarSquares, NC);
        else wait_cluster(mbar + 2 + buf);
        // lane l adds up slice l % 8 of token l / 16 (of two), or slice l % 16, then they add up each other's: one load and one root per lane
        constexpr int R = NW > 8 ? 16 : 8;
        const int from = lane & (R - 1);
        const uint4 part = lds128(sq + static_cast<uint32_t>((T == 2 ? lane >> 4 : 0) * NW + (from < NW ? from : 0)) * 16u);
        float total = (__uint_as_float(part.x) + __uint_as_float(part.y)) + (__uint_as_float(part.z) + __uint_as_float(part.w));
        if (from >= NW) total = 0.f;
#pragma unroll
        for (int o = R / 2; o >= 1; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
        float mean = total * (1.0f / D);
        if constexpr ((D & (D - 1)) != 0)  // the correctly rounded quotient (an infinite total would make the correction NaN)
            mean = total < INFINITY ? fmaf(fmaf(-mean, static_cast<float>(D), total), 1.0f / D, mean) : total;
        const float own = rsqrt_refined(mean + eps);
#pragma unroll
        for (int j = 0; j < T; ++j) {
            const float r = T == 2 ? __shfl_sync(0xffffffffu, own, 16 * j) : own;
#pragma unroll
            for (int i = 0; i < 4; ++i) sts16(normed + static_cast<uint32_t>(j) * 256u + own_off + col(i), float_to_bf16_bits((h[j][i] * r) * bf16_bits_to_float(w[i])));
        }
        __syncwarp();
    }
    // this warp's partial logits
    __device__ __forceinline__ void logits(const RouterA<N> &w, uint32_t buf)
    {
        float z[N / 16][4];
        w.product((NORM ? normed : hid) + b_off, z);
        const int r = lane >> 2, q = lane & 3;  // columns 2q, 2q + 1 of the product; token 0's are 0 - 3
        if constexpr (CS == 1) {
            if (q == 0 || (T == 2 && q == 2)) {
                const uint32_t at = partial + (buf * NW + static_cast<uint32_t>(warp)) * (T * N * 4u) + static_cast<uint32_t>((T == 2 ? q >> 1 : 0) * N + r) * 4u;
                stsf(at, z[0][0]);
                stsf(at + 32u, z[0][2]);
            }
        } else if constexpr (CS == 2) {  // all columns are equal: lane q pushes to block q / 2, experts r or 8 + r
            static_assert(N == 16, "four lanes have an expert's logit");
            const uint32_t at = partial + (buf * NW + static_cast<uint32_t>(slice)) * (N * 4u) + static_cast<uint32_t>(r + 8 * (q & 1)) * 4u, to = static_cast<uint32_t>(q) >> 1;
            cluster_push_f32(cluster_map(at, to), (q & 1) ? z[0][2] : z[0][0], cluster_map(smem_u32(mbar + buf), to));
        } else {  // ... to block q, every expert it has
            static_assert(CS == 4, "four lanes have an expert's logit");
            const uint32_t at = cluster_map(partial + (buf * NW + static_cast<uint32_t>(slice)) * (N * 4u) + static_cast<uint32_t>(r) * 4u, q);
            const uint32_t bar = cluster_map(smem_u32(mbar + buf), q);
#pragma unroll
            for (int i = 0; i < N / 8; ++i) cluster_push_f32(at + 32u * i, z[i >> 1][2 * (i & 1)], bar);
        }
    }
    // softmax numerators (Eq. 4): lane 16 j + e has token j's expert e (one token of 16: both halves have it).  `loads`: what is to be
    // asked of shared memory while the numerators and the weighted sum are computed -- not before, where the partial logits and
    // the state would queue behind it
    template <typename F>
    __device__ __forceinline__ float numerators(uint32_t buf, F &&loads)
    {
        if constexpr (CS == 1) named_bar_sync(kBarLogits, COUNT);
        else wait_cluster(mbar + buf);
        const uint32_t at = partial + buf * static_cast<uint32_t>(NW * T * N * 4) + static_cast<uint32_t>(T == 2 || N == 32 ? lane : lane & 15) * 4u;
        float v[NW];
#pragma unroll
        for (int i = 0; i < NW; ++i) v[i] = ldsf(at + static_cast<uint32_t>(i) * (T * N * 4u));
        loads();
        float even = v[0], odd = v[1];
#pragma unroll
        for (int i = 2; i < NW; i += 2) even += v[i], odd += v[i + 1];
        return softmax_part(even + odd, N);
    }
    // weighted sum (Eq. 8), residual, one rounding: the new state, in registers and in the hidden slices.  after(j): token j's rows
    // have been given to the product
    template <typename F>
    __device__ __forceinline__ void weighted(const RowsA<N> (&rows)[T], float e, const bool (&valid)[T], F &&after)
    {
        GateColumns<N> g[T];
#pragma unroll
        for (int j = 0; j < T; ++j) g[j].from_lanes(e, lane, 16 * j);
#pragma unroll
        for (int j = 0; j < T; ++j) {
            float v[4], inv;
            rows[j].product(g[j], lane, v, [&]() {
                inv = __frcp_rn(g[j].sum());
                after(j);
            });
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const unsigned short o = float_to_bf16_bits(valid[j] ? fmaf(v[i], inv, h[j][i]) : h[j][i]);
                h[j][i] = bf16_bits_to_float(o);
                sts16(hid + static_cast<uint32_t>(j) * 256u + own_off + col(i), o);
            }
        }
        __syncwarp();
    }
};

__device__ __forceinline__ long long slice_id(const StepParams &p, long long t)
{
    return (p.flags & MOLE_FLAG_IDS_INT64) ? __ldg(static_cast<const long long *>(p.row_index) + t)
                                           : static_cast<long long>(__ldg(static_cast<const int *>(p.row_index) + t));
}

// The fused step: a block walks its groups of T tokens (group b, b + G, ..) through the L layers; (group, layer) is an item.  Slot
// i % S holds item i's rows and router matrix, copied as one group or, of 32 experts, as two: they are large, it is the rows that come from
// DRAM, and so they need not have landed as early as the matrix (16 layers, 16 tokens: 18.2 us).
// Which wait covers which read (i: an item; its barrier is the one its partial logits are counted in at):
//   - Landed.  What a compute warp reads behind barrier i has landed before the copying warps arrive at it; what it reads ahead of
//     barrier i -- a cluster's warps, under the exchange -- has landed before barrier i - 1.  One block: item i + 1 behind barrier i.  Clusters:
//     the matrix of item i + 1 ahead of barrier i, and its rows there, too (16 experts) or behind it (32).
//   - Overwritten.  Behind barrier i the copying warps fill the slot of item i with item i + S.  A compute warp asks for item i's rows and
//     matrix ahead of or just behind barrier i - 1, and later gives its partial logits of item i to barrier i.  One block: barrier i is
//     a block barrier.  Clusters: those logits are computed from the matrix itself and from a state that was read from shared memory
//     after the rows, and a warp's shared-memory requests are served in order.
template <int N, int D, int T, int NORM, int CS>
__global__ void __cluster_dims__(CS, 1, 1) __launch_bounds__((D / kMmaCols / CS + slice_copy_warps(N)) * 32, 1) mole_slice_step_kernel(const StepParams p)
{
    constexpr int NW = D / kMmaCols / CS, S = slice_slots(N, NW, T, CS), kCopyWarps = slice_copy_warps(N);  // warps of this block
    // groups of copies per item; how many may be on their way when the first item is read, and at a barrier
    constexpr int GROUPS = N == 32 ? 2 : 1, FIRST_PENDING = S * GROUPS - (CS == 1 ? 1 : GROUPS == 2 ? 3 : 2),
                  PENDING = GROUPS == 2 ? 1 : S - (CS == 1 ? 2 : 3);
    static_assert(FIRST_PENDING >= 0 && PENDING >= 0, "slots");
    static_assert(CS == 1 ? 2 <= S - PENDING                           // behind barrier i: item i + 1, of the S + i copied by then
                          : GROUPS == 1 ? 3 <= S - PENDING             // ahead of it: item i + 1, of the S + i - 1 behind barrier i - 1
                                        : 5 <= 2 * S - PENDING,            // its matrix; one group less for its rows, behind barrier i
                  "copies that are read have landed");
    using Layer = SliceLayer<N, D, T, NORM, (NW + kCopyWarps) * 32, CS>;
    constexpr SliceSmem m = slice_smem(N, NW, T, S, NORM, CS);
    constexpr uint32_t kRows = NW * slice_bytes(N);  // of a slot: the router matrix, then the rows
    extern __shared__ __align__(1024) unsigned char smem_1k[];
    unsigned char *const smem = smem_1k;

    pdl_enter(p.flags);

    const uint32_t base = smem_u32(smem);
    const int lane = static_cast<int>(threadIdx.x) & 31, warp = static_cast<int>(threadIdx.x) >> 5, L = p.L;
    const uint32_t rank = CS > 1 ? cluster_ctarank() : 0u;
    const long long G = gridDim.x / CS, g0 = blockIdx.x / CS, groups = (p.M + T - 1) / T;
    uint64_t *mbar = reinterpret_cast<uint64_t *>(smem + m.off_bar);
    volatile int *dead = reinterpret_cast<volatile int *>(mbar + 4);
    if constexpr (CS > 1) {
        if (threadIdx.x == 0) {
            for (int i = 0; i < 4; ++i) mbar_init(mbar + i, i < 2 ? 1 + kCopyWarps : 1);
            dead[0] = 0;
            mbar_init_fence();
        }
        __syncthreads();
        cluster_arrive();  // waited for before the first push
    }

    if (warp >= NW) {
        // ================= copying warps: warp NW + k copies the slices k, k + kCopyWarps, .. =================
        const int first = warp - NW;
        const unsigned char *w0 = static_cast<const unsigned char *>(p.w_router) + rank * (NW * slice_bytes(N)), *w = w0;
        const unsigned char *row[T];
        long long g = g0, next_id[T], gw = g0;  // the group whose rows are issued next; ids of the group after; the routers' group
        int l = 0, s = 0, lw = 0, sw = 0;
        auto fetch_ids = [&](long long gg) {
#pragma unroll
            for (int j = 0; j < T; ++j) next_id[j] = gg < groups && gg * T + j < p.M ? slice_id(p, gg * T + j) : -1;
        };
        auto begin_group = [&]() {
#pragma unroll
            for (int j = 0; j < T; ++j) {
                const bool ok = next_id[j] >= 0 && next_id[j] < p.rows;  // otherwise row 0 is fetched and its term dropped
                row[j] = static_cast<const unsigned char *>(p.lut) + static_cast<size_t>(ok ? next_id[j] : 0) * (N * D * 2) + rank * (NW * 256u);
            }
            fetch_ids(g + G);
        };
        auto router = [&]() {  // the next router matrix
            if (gw >= groups) return;
#pragma unroll
            for (int c0 = 0; c0 < NW; c0 += kCopyWarps) {
                const int c = c0 + first;
                if (NW % kCopyWarps == 0 || c < NW) slice_copy_router<N>(base + static_cast<uint32_t>(sw) * m.slot + static_cast<uint32_t>(c) * slice_bytes(N), w + c * slice_bytes(N), lane);
            }
            w += p.wr_stride;
            if (++lw == L) lw = 0, gw += G, w = w0;
            if (++sw == S) sw = 0;
        };
        auto token_rows = [&]() {  // the next item's rows
            if (g >= groups) return;
#pragma unroll
            for (int j = 0; j < T; ++j) {
#pragma unroll
                for (int c0 = 0; c0 < NW; c0 += kCopyWarps) {
                    const int c = c0 + first;
                    if (NW % kCopyWarps == 0 || c < NW)
                        slice_copy_rows<N, D>(base + static_cast<uint32_t>(s) * m.slot + kRows + static_cast<uint32_t>(j * NW + c) * slice_bytes(N), row[j] + c * 256, lane);
                }
                row[j] += p.lut_stride;
            }
            if (++l == L) {
                l = 0;
                g += G;
                begin_group();
            }
            if (++s == S) s = 0;
        };
        auto issue = [&]() {  // the next item's groups of copies (empty ones behind the last item)
            router();
            if constexpr (GROUPS == 2) cp_async_commit();
            token_rows();
            cp_async_commit();
        };
        fetch_ids(g);
        begin_group();
#pragma unroll 1
        for (int i = 0; i < S; ++i) issue();
        cp_async_wait<FIRST_PENDING>();
        __syncthreads();  // what is read ahead of item 0's barrier has landed
        Layer y;
        if constexpr (CS > 1) {
            y.init(base, m);
            y.mbar = mbar, y.dead = dead, y.status = p.status, y.polls = p.wait_polls;
        }
        uint32_t buf = 0;
        for (long long gg = g0; gg < groups; gg += G)
            for (int i = 0; i < L; ++i) {
                cp_async_wait<PENDING>();
                if constexpr (CS == 1) {
                    named_bar_sync(Layer::kBarLogits, Layer::COUNT);
                } else {
                    __syncwarp();
                    if (lane == 0 && y.alive) mbar_arrive(mbar + buf);
                    y.wait_cluster(mbar + buf);
                    __syncwarp();
                    buf ^= 1u;
                    if (buf == 0) y.phase ^= 1u;
                }
                issue();
            }
        cp_async_wait<0>();
        if constexpr (CS > 1) {
            __syncwarp();
            cluster_wait();
            cluster_arrive();
            cluster_wait();
        }
        return;
    }

    Layer y;
    y.init(base, m);
    y.mbar = mbar, y.dead = dead, y.status = p.status, y.polls = p.wait_polls;
    const unsigned char *norm_g = static_cast<const unsigned char *>(p.norm_weight) + y.slice * 256 + y.own_off;
    unsigned short wgt[4] = {0, 0, 0, 0};  // as loaded: whatever is done to them here would wait for them here
    auto load_norm = [&](int l) {
#pragma unroll
        for (int i = 0; i < 4; ++i) wgt[i] = __ldg(reinterpret_cast<const unsigned short *>(norm_g + static_cast<size_t>(l) * p.norm_stride + Layer::col(i)));
    };
    if constexpr (NORM) load_norm(0);
    RouterA<N> wf;
    wf.init(lane);
    const uint32_t w_lane = static_cast<uint32_t>(warp) * slice_bytes(N), r_lane = w_lane + RowsA<N>::lane_offset(lane);
    RowsA<N> rows[T];
    uint32_t buf = 0;
    int s = 0;
    auto load_rows = [&](RowsA<N> &r, int j) { r.load(base + static_cast<uint32_t>(s) * m.slot + kRows + static_cast<uint32_t>(j * NW) * slice_bytes(N) + r_lane); };
    __syncthreads();
    wf.load(base + w_lane);
#pragma unroll
    for (int j = 0; j < T; ++j) load_rows(rows[j], j);
    if constexpr (CS > 1) cluster_wait();

    pdl_wait();

#pragma unroll 1
    for (long long g = g0; g < groups; g += G) {
        bool valid[T];
#pragma unroll
        for (int j = 0; j < T; ++j) {
            const long long id = g * T + j < p.M ? slice_id(p, g * T + j) : -1;
            valid[j] = id >= 0 && id < p.rows;
            if (!valid[j] && g * T + j < p.M && threadIdx.x == 0 && rank == 0 && p.status) atomicOr(p.status, MOLE_STATUS_BAD_ID);
        }
        y.load_hidden(static_cast<const unsigned char *>(p.hidden), g * T, p.M, []() {});
#pragma unroll(T == 1 && N == 16 ? 2 : 1)
        for (int l = 0; l < L; ++l) {
            y.arm(buf);
            if constexpr (NORM) {
                y.normalise(wgt, p.norm_eps, buf);
                load_norm(l + 1 < L ? l + 1 : 0);
            }
            y.logits(wf, buf);
            if (++s == S) s = 0;
            // one token: the next rows go to registers of their own; two tokens: to those of the rows just multiplied
            RowsA<N> next;
            if constexpr (CS > 1) {  // the exchange is long enough to hide both (32 experts: to hide one, and the registers for one)
                wf.load(base + static_cast<uint32_t>(s) * m.slot + w_lane);
                if constexpr (N == 16) load_rows(next, 0);
            }
            const float e = y.numerators(buf, [&]() {
                if constexpr (CS == 1) wf.load(base + static_cast<uint32_t>(s) * m.slot + w_lane);
            });
            y.weighted(rows, e, valid, [&](int j) {
                if constexpr (CS == 1 || N == 32) load_rows(T == 1 && N == 16 ? next : rows[j], j);
            });
            if constexpr (T == 1 && N == 16) rows[0] = next;
            buf ^= 1u;
            if (CS > 1 && buf == 0) y.phase ^= 1u;
        }
        y.store_out(static_cast<unsigned char *>(p.out), g * T, p.M);
    }
    if constexpr (CS > 1) {
        if (!y.alive)  // the other block's pushes have not been waited for: time to land, before the blocks can exit
            for (int i = 0; i < 32; ++i) __nanosleep(1000);
        __syncwarp();
        cluster_arrive();  // nobody leaves before everybody is done
        cluster_wait();
    }
}

// One layer, a block per group of T tokens.  What does not depend on the kernel before -- router matrix (one bulk copy for the
// block), rows -- is requested before it is waited for.  LOOP: a launch of more groups than are resident at once; a block then walks every
// gridDim.x-th, and copies the rows of the next into the slots as soon as it has those of this one in registers: where 300 groups met
// 296 places the last four cost a wave of their own (chained layers, us each, a block per group / here: 16 x 1024, 600 tokens 6.1 / 4.7, with the
// norm 7.1 / 6.0; 888 tokens 6.9 / 5.7, 8.0 / 6.8; 16 x 768, 600 tokens 5.0 / 3.7, 5.8 / 4.4).
template <int LOOP>
struct SliceIndex {
    using type = int;
};
template <>
struct SliceIndex<0> {
    using type = long long;
};
template <int D, int T, int NORM, int LOOP>
__global__ void __launch_bounds__(D / kMmaCols * 32, 2) mole_slice_layer_kernel(const StepParams p)
{
    constexpr int N = 16, NW = D / kMmaCols;
    using Layer = SliceLayer<N, D, T, NORM, NW * 32>;
    constexpr SliceSmem m = slice_smem(N, NW, T, 1, NORM);
    constexpr uint32_t kRouterBytes = D * N * 2;
    extern __shared__ __align__(1024) unsigned char smem_1k[];
    unsigned char *const smem = smem_1k;

    pdl_enter(p.flags);

    const uint32_t base = smem_u32(smem);
    Layer y;
    y.init(base, m);
    const int lane = y.lane, warp = y.warp;
    // (a launch has fewer than 2^30 tokens; without the loop 64 bits measured 1 - 2 % faster, with it they are spilled)
    using Index = typename SliceIndex<LOOP>::type;
    const Index M = static_cast<Index>(p.M);
    Index t0 = static_cast<Index>(blockIdx.x) * T;
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + m.off_bar);
    volatile int *dead = reinterpret_cast<volatile int *>(bar + 1);
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        dead[0] = 0;
        dead[1] = 0;  // raised by nobody: lets the drain wait run its (short) course
        mbar_init_fence();
        mbar_expect_tx(bar, kRouterBytes);
        bulk_g2s(smem, p.w_router, kRouterBytes, bar);
    }
    bool valid[T], valid_next[T];  // of the tokens at hand; of those whose rows are on their way
    const uint32_t slots = base + static_cast<uint32_t>(NW + warp) * slice_bytes(N);  // this warp's slices, one per token
    auto copy_rows = [&](Index t1) {
        long long id[T];
#pragma unroll
        for (int j = 0; j < T; ++j) id[j] = t1 + j < M ? slice_id(p, t1 + j) : -1;
#pragma unroll
        for (int j = 0; j < T; ++j) {
            valid_next[j] = id[j] >= 0 && id[j] < p.rows;  // otherwise row 0 is fetched and its term dropped
            const unsigned char *row = static_cast<const unsigned char *>(p.lut) + static_cast<size_t>(valid_next[j] ? id[j] : 0) * (N * D * 2) + warp * 256;
            slice_copy_rows<N, D>(slots + static_cast<uint32_t>(j) * (NW * slice_bytes(N)), row, lane);
            if (!valid_next[j] && t1 + j < M && threadIdx.x == 0 && p.status) atomicOr(p.status, MOLE_STATUS_BAD_ID);
        }
        cp_async_commit();
    };
    copy_rows(t0);
    __syncthreads();  // the barrier is initialised
    if (!wait_or_give_up(bar, 0, dead, p.wait_polls)) {  // nothing waits any more: what is there is computed on, and the status says so
        if (lane == 0) report_timeout(dead, p.status);
        (void)wait_or_give_up(bar, 0, dead + 1, kDrainPolls);
    }
    // the matrix lies as it does in memory, 32 bytes a column: two-way bank conflicts, but ahead of the wait for the kernel before
    RouterA<N> wf;
    {
        const uint32_t w = base + static_cast<uint32_t>(warp) * slice_bytes(N) + static_cast<uint32_t>(8 * (lane >> 4) + (lane & 7)) * 32u + static_cast<uint32_t>((lane >> 3) & 1) * 16u;
#pragma unroll
        for (int k = 0; k < 8; ++k) ldsm_x4_trans(wf.a[k][0], w + static_cast<uint32_t>(k) * 512u);
    }
    uint32_t buf = 0;
#pragma unroll 1
    for (bool first = true;; first = false) {
        cp_async_wait<0>();
        __syncwarp();
        RowsA<N> rows[T];
#pragma unroll
        for (int j = 0; j < T; ++j) rows[j].load(slots + static_cast<uint32_t>(j) * (NW * slice_bytes(N)) + RowsA<N>::lane_offset(lane));
#pragma unroll
        for (int j = 0; j < T; ++j) valid[j] = valid_next[j];
        const Index t1 = t0 + static_cast<Index>(gridDim.x) * T;
        const bool more = LOOP != 0 && t1 < M;
        if (LOOP) {
            __syncwarp();
            if (more) copy_rows(t1);
        }

        if (first) pdl_wait();

        uint32_t wgt[4] = {0u, 0u, 0u, 0u};
        unsigned short res[T][4] = {};
        auto load_residual = [&]() {
            if (!p.residual) return;
            const unsigned char *src = static_cast<const unsigned char *>(p.residual) + warp * 256 + y.own_off;
#pragma unroll
            for (int j = 0; j < T; ++j)
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (t0 + j < M) res[j][i] = __ldcg(reinterpret_cast<const unsigned short *>(src + static_cast<size_t>(t0 + j) * (D * 2) + Layer::col(i)));
        };
        if (!LOOP) load_residual();
        y.load_hidden(static_cast<const unsigned char *>(p.hidden), t0, M, [&]() {
            if constexpr (NORM) {  // MOLE_FLAG_CHAIN does not forbid the kernel before to write the scale
#pragma unroll
                for (int i = 0; i < 4; ++i) wgt[i] = ld_scale_u16(static_cast<const unsigned char *>(p.norm_weight) + warp * 256 + y.own_off + Layer::col(i));
            }
        });
        if constexpr (NORM) y.normalise(wgt, p.norm_eps, buf);
        y.logits(wf, buf);
        auto use_residual = [&]() {  // it takes the hidden state's place in what follows
            if (!p.residual) return;
#pragma unroll
            for (int j = 0; j < T; ++j)
#pragma unroll
                for (int i = 0; i < 4; ++i) y.h[j][i] = bf16_bits_to_float(res[j][i]);
        };
        if (LOOP) load_residual();  // (late, for want of registers)
        else use_residual();
        const float e = y.numerators(buf, []() {});
        if (LOOP) use_residual();
        if (p.gates_out && warp == 0) {
            float sum = e;
#pragma unroll
            for (int o = 8; o >= 1; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            const Index t = t0 + (T == 2 ? lane >> 4 : 0);
            if ((T == 2 || lane < 16) && t < M) p.gates_out[static_cast<size_t>(t) * N + (lane & 15)] = e / sum;
        }
        y.weighted(rows, e, valid, [](int) {});
        y.store_out(static_cast<unsigned char *>(p.out), t0, M);
        if (!more) break;
        t0 = t1;
        buf ^= 1u;
        __syncwarp();  // the state has been stored: its slices are free
    }
}

#endif  // __CUDACC__

}  // namespace mole
