// The prefill form of the fused MoLE layer for sm_100a (Eq. 4 and Eq. 8 of arXiv 2503.15798): one layer, many tokens, bf16,
// N of 8, 16 or 32 experts, d a multiple of 128 up to 2048.
//
// What bounds it.  A token is N d multiply-adds for the router and as many for the weighted sum, over rows that come from
// L2 or DRAM once: at thousands of tokens the launch is bound by issue slots first (the ring kernel spends 3 200 warp
// instructions per token of the 410M shape) and by the latency and the rows' way into the SMs second.  So:
//   - Router on the tensor cores: the block walks over groups of tb tokens; warp w multiplies the group's hidden states by
//     its 128 rows of the router matrix (mma.m16n8k16: rows of A are tokens, bf16 products, fp32 sums).  The matrix stays in
//     shared memory for the whole launch, in 16-byte pieces swizzled for conflict-free ldmatrix; the next group's hidden
//     states are copied in (cp.async) under this group's sums.
//   - One meeting per group: the partial logits of all warps.  From there on a warp owns a token (or half of its columns):
//     it sums the partials, forms the softmax numerators and accumulates the token's rows, which go straight from global
//     memory into registers, 16 bytes per lane, one batch of experts in flight while another is accumulated (packed fp32
//     fmas, experts in ascending order).  The first rows of a warp's next token are requested before its turn comes.
// Measured, calls back to back, ring kernel / here, us: 16 384 tokens of the 410M shape 88.2 / 53.1 (with the norm 98.5 / 60.5), of the
// 160M shape 69.7 / 40.3 (89.1 / 46.9); 2 999 tokens of the 1B shape with the norm and a residual 78.9 / 47.9; 4 000 tokens of 32 x 1024
// 96.3 / 33.3; 8 000 of 8 x 512 24.7 / 14.2.  At 410M one launch moves 635 MB into the SMs (537 of them rows) at 11.5 TB/s and 209 MB
// out of DRAM at 0.58 of the copy rate; issue slots are 48 % busy, L2 44 %, L1 63 %.  No unit is full: the 22 warps an SM has at 80
// registers wait for rows (5.4 long-scoreboard stalls per issue).  Batches of four experts in 80 registers (three blocks per SM)
// against eight in 128 (two): 54 and 57 us at d = 1024, 41 and 52 us at 768.  Tried and slower: an L2 prefetch of the next token's
// rows (57 -> 67 us); 24 warps around one resident matrix (64 us); the weighted sum on the tensor cores with the numerators cut
// into bf16 parts, rows through shared memory (108 us).
// The order of every fp32 sum is fixed by N and d: a token gets the same bits in any batch this kernel runs.
#pragma once

#include "mole_decode.cuh"

namespace mole {

constexpr int kSliceCols = 128;   // columns of a warp's router slice
constexpr int kTileMaxWarps = 16;
constexpr int kHidStride = 272;   // bytes between two tokens' hidden slices: 256 + 16, so that eight rows of an ldmatrix hit different banks
// Width classes: d itself where it is compiled in (the widths of Table 2), any d up to 1024, any d up to 2048.
constexpr int kTileNarrow = -1, kTileWide = 0;
__host__ __device__ constexpr bool tile_narrow(int D) { return D == kTileNarrow || (D > 0 && D <= 1024); }

struct TileParams {
    const void *hidden, *residual, *row_index, *lut, *w_router, *norm_weight;
    void *out;
    float *gates_out;
    uint32_t *status;
    long long M, rows;
    int d;
    int tb;  // tokens per group (at most 16)
    int groups;
    float norm_eps;
    uint32_t flags;
};

// router matrix, hidden slices, partial logits, softmax numerators, sums of squares
struct TileSmem {
    uint32_t off_hid, off_partial, off_gates, off_ssq, total;
};
__host__ __device__ inline TileSmem tile_smem(int N, int d, int tb, int norm)
{
    TileSmem m;
    const int warps = d / kSliceCols;
    m.off_hid = static_cast<uint32_t>(d) * N * 2;
    m.off_partial = m.off_hid + static_cast<uint32_t>(warps * tb * kHidStride);
    m.off_gates = m.off_partial + static_cast<uint32_t>(tb * warps * N * 4);
    m.off_ssq = m.off_gates + static_cast<uint32_t>(warps * N * 4);
    m.total = m.off_ssq + (norm ? static_cast<uint32_t>(tb * warps * 4) : 0u);
    return m;
}

#ifdef __CUDACC__

__device__ __forceinline__ uint4 ldg_stream_v4(const void *p)
{
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
// Position of 16-byte piece c of row k of a router slice [rows][N]: eight consecutive rows of one piece (an ldmatrix phase)
// fall into eight different 16-byte bank groups.
template <int N>
__device__ __forceinline__ uint32_t router_piece(int k, int c)
{
    if constexpr (N == 8) return static_cast<uint32_t>(k);
    else if constexpr (N == 16) return static_cast<uint32_t>(2 * k + (c ^ ((k >> 2) & 1)));
    else return static_cast<uint32_t>(4 * k + (c ^ ((k >> 1) & 3)));
}
// four bf16 times r times four scale entries, rounded once
__device__ __forceinline__ uint2 scale_bf16x4(uint2 h, float r, float w0, float w1, float w2, float w3)
{
    const __nv_bfloat162 lo = __floats2bfloat162_rn((bf16_bits_to_float(h.x & 0xffffu) * r) * w0, (__uint_as_float(h.x & 0xffff0000u) * r) * w1);
    const __nv_bfloat162 hi = __floats2bfloat162_rn((bf16_bits_to_float(h.y & 0xffffu) * r) * w2, (__uint_as_float(h.y & 0xffff0000u) * r) * w3);
    return make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
}
__device__ __forceinline__ float sum_squares4(uint2 h)
{
    const float x0 = bf16_bits_to_float(h.x & 0xffffu), x1 = __uint_as_float(h.x & 0xffff0000u);
    const float x2 = bf16_bits_to_float(h.y & 0xffffu), x3 = __uint_as_float(h.y & 0xffff0000u);
    return fmaf(x3, x3, fmaf(x2, x2, fmaf(x1, x1, x0 * x0)));
}

// N: experts.  NORM: the router reads RMSNorm(hidden).  D: width class.  PARTS: warps per token (each takes d / PARTS columns);
// a constant because the column arithmetic of a run-time one costs 20 % at d = 1024.
// Launch: d / 4 threads, tile_smem(..).total bytes, any grid.
template <int N, int NORM, int D, int PARTS>
__global__ void __launch_bounds__(tile_narrow(D) ? 256 : kTileMaxWarps * 32, tile_narrow(D) ? 3 : 1) mole_tile_kernel(const TileParams p)
{
    constexpr int NT = N / 8;
    constexpr int SLICE = kSliceCols * N * 2;
    constexpr int EB = tile_narrow(D) || N == 8 ? 4 : 8;  // experts per load batch
    constexpr int BATCHES = N / EB;
    extern __shared__ __align__(128) unsigned char smem[];

    pdl_enter(p.flags);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int d = D > 0 ? D : p.d, nw = d / kSliceCols;
    const int TB = p.tb;
    const TileSmem m = tile_smem(N, d, TB, NORM);
    const uint32_t base = smem_u32(smem);
    const uint32_t w_s = base + static_cast<uint32_t>(warp) * SLICE;
    const uint32_t hid_own = m.off_hid + static_cast<uint32_t>(warp * TB * kHidStride);
    float *partial = reinterpret_cast<float *>(smem + m.off_partial);  // [TB][nw][N]
    float *gates = reinterpret_cast<float *>(smem + m.off_gates) + warp * N;
    float *ssq = reinterpret_cast<float *>(smem + m.off_ssq);          // [TB][nw]
    const bool ids64 = (p.flags & MOLE_FLAG_IDS_INT64) != 0;
    const int G = gridDim.x, b0 = blockIdx.x;
    const int wt = warp / PARTS, part = warp - wt * PARTS;  // this warp's tokens of a group: wt, wt + nw / PARTS, ...
    const int wstep = nw / PARTS;
    const int cols = d / PARTS;
    const int npass = (cols + 255) >> 8;

    // the router matrix slice, once
    {
        const unsigned char *src = static_cast<const unsigned char *>(p.w_router) + static_cast<size_t>(warp) * SLICE + lane * 16;
        const uint32_t dst = w_s + 16u * (N == 8 ? lane : (N == 16 ? router_piece<16>(lane >> 1, lane & 1) : router_piece<32>(lane >> 2, lane & 3)));
#pragma unroll
        for (int c = 0; c < SLICE / 512; ++c) cp_async16(dst + 512u * c, src + 512 * c);
    }
    auto id_of = [&](long long t) -> long long {
        return ids64 ? __ldg(static_cast<const long long *>(p.row_index) + t) : static_cast<long long>(__ldg(static_cast<const int *>(p.row_index) + t));
    };
    // the sequence of this warp's tokens: (group, wt), (group, wt + wstep), ..., the next group, ...; -1 after the last
    auto next_token = [&](int &g, int &k) -> long long {
        k += wstep;
        if (k >= TB) {
            k = wt;
            g += G;
        }
        const long long t = static_cast<long long>(g) * TB + k;
        return g < p.groups && k < TB && t < p.M ? t : -1;
    };
    const size_t row_bytes = static_cast<size_t>(N) * d * 2;
    const size_t lane_off = static_cast<size_t>(part) * cols * 2 + lane * 16;
    uint4 ra[EB], rb[EB];
    auto load = [&](uint4 (&r)[EB], const unsigned char *row, int pass, int batch, bool on) {
        // (lanes past the last column re-read the row's first vector)
        const unsigned char *src = row + static_cast<size_t>(batch * EB) * d * 2 + (pass * 256 + lane * 8 < cols ? pass * 512 : -static_cast<int>(lane_off));
        if (on) {
#pragma unroll
            for (int j = 0; j < EB; ++j) r[j] = ldg_stream_v4(src + static_cast<size_t>(j) * d * 2);
        }
    };
    int g_next = b0, k_next = wt - wstep;
    long long t_next = next_token(g_next, k_next);
    long long id_next = t_next >= 0 ? id_of(t_next) : -1;
    bool v_next = id_next >= 0 && id_next < p.rows;
    const unsigned char *row_next = static_cast<const unsigned char *>(p.lut) + static_cast<size_t>(v_next ? id_next : 0) * row_bytes + lane_off;
    load(ra, row_next, 0, 0, v_next);

    pdl_wait();

    // this warp's hidden slices of group g
    auto fetch_hidden = [&](int g) {
        if (g < p.groups) {
            const unsigned char *src = static_cast<const unsigned char *>(p.hidden) + static_cast<size_t>(warp) * (kSliceCols * 2) + (lane & 15) * 16;
            const uint32_t dst = base + hid_own + (lane & 15) * 16;
            for (int k = lane >> 4; k < TB; k += 2) {
                long long t = static_cast<long long>(g) * TB + k;
                if (t >= p.M) t = p.M - 1;  // rows past the last token repeat it; nothing of them is used
                cp_async16(dst + static_cast<uint32_t>(k * kHidStride), src + static_cast<size_t>(t) * d * 2);
            }
        }
        cp_async_commit();
    };
    fetch_hidden(b0);

#pragma unroll 1
    for (int g = b0; g < p.groups; g += G) {
        cp_async_wait_all();
        __syncwarp();
        const uint32_t hid = base + hid_own;
        if constexpr (NORM) {
            // y = (x / sqrt(mean(x^2) + eps)) * w, rounded once to bf16, in place; eight tokens at a time
            unsigned char *hl = smem + hid_own + lane * 8;
            for (int k0 = 0; k0 < TB; k0 += 8) {
                float s[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) s[k] = sum_squares4(*reinterpret_cast<const uint2 *>(hl + (k0 + k < TB ? k0 + k : TB - 1) * kHidStride));
                int first = 0;
                lane_reduce_scatter<8, 8, 16, 1>(s, lane, first);
                if ((lane & 3) == 0 && k0 + first < TB) ssq[(k0 + first) * nw + warp] = s[0];
            }
            const uint2 wv = ld_scale_v2(static_cast<const unsigned char *>(p.norm_weight) + static_cast<size_t>(warp) * (kSliceCols * 2) + lane * 8);
            __syncthreads();
            const float w0 = bf16_bits_to_float(wv.x & 0xffffu), w1 = __uint_as_float(wv.x & 0xffff0000u);
            const float w2 = bf16_bits_to_float(wv.y & 0xffffu), w3 = __uint_as_float(wv.y & 0xffff0000u);
            float total = 0.f;
            const float *sq = ssq + (lane < TB ? lane : 0) * nw;
            for (int w = 0; w < nw; ++w) total += sq[w];  // slices in ascending order
            const float rinv = rms_scale(total, d, p.norm_eps);
            for (int k = 0; k < TB; ++k) {
                const float r = __shfl_sync(0xffffffffu, rinv, k);
                uint2 *x = reinterpret_cast<uint2 *>(hl + k * kHidStride);
                *x = scale_bf16x4(*x, r, w0, w1, w2, w3);
            }
            __syncwarp();
        }

        // ---- router: partial logits of the group's tokens over this warp's columns, steps of 16 columns in two chains ----
        float acc[NT][4], odd[NT][4];
        {
            const int i = lane & 7, mm = lane >> 3;
            const int row = i + 8 * (mm & 1);
            const uint32_t a_addr = hid + static_cast<uint32_t>((row < TB ? row : TB - 1) * kHidStride + (mm >> 1) * 16);
#pragma unroll
            for (int t = 0; t < NT; ++t)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[t][e] = odd[t][e] = 0.f;
#pragma unroll
            for (int s = 0; s < kSliceCols / 16; s += 2) {
                uint32_t a0[4], a1[4];
                ldsm_x4(a0, a_addr + 32u * s);
                ldsm_x4(a1, a_addr + 32u * s + 32u);
                if constexpr (N == 8) {
                    uint32_t b[4];
                    ldsm_x4_trans(b, w_s + 16u * router_piece<N>(16 * s + 8 * mm + i, 0));
                    mma16(acc[0], a0[0], a0[1], a0[2], a0[3], b[0], b[1]);
                    mma16(odd[0], a1[0], a1[1], a1[2], a1[3], b[2], b[3]);
                } else {
#pragma unroll
                    for (int q = 0; q < NT / 2; ++q) {
                        uint32_t b[4], c[4];
                        const int k = 16 * s + 8 * (mm & 1) + i, piece = 2 * q + (mm >> 1);
                        ldsm_x4_trans(b, w_s + 16u * router_piece<N>(k, piece));
                        ldsm_x4_trans(c, w_s + 16u * router_piece<N>(k + 16, piece));
                        mma16(acc[2 * q], a0[0], a0[1], a0[2], a0[3], b[0], b[1]);
                        mma16(acc[2 * q + 1], a0[0], a0[1], a0[2], a0[3], b[2], b[3]);
                        mma16(odd[2 * q], a1[0], a1[1], a1[2], a1[3], c[0], c[1]);
                        mma16(odd[2 * q + 1], a1[0], a1[1], a1[2], a1[3], c[2], c[3]);
                    }
                }
            }
        }
        if (g != b0) named_bar_sync(1, 2 * nw * 32);  // the previous group's partials have been read by everybody
        {
            const int r = lane >> 2, q = lane & 3;
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                if (r < TB) *reinterpret_cast<float2 *>(partial + (r * nw + warp) * N + 8 * t + 2 * q) = make_float2(acc[t][0] + odd[t][0], acc[t][1] + odd[t][1]);
                if (r + 8 < TB) *reinterpret_cast<float2 *>(partial + ((r + 8) * nw + warp) * N + 8 * t + 2 * q) = make_float2(acc[t][2] + odd[t][2], acc[t][3] + odd[t][3]);
            }
        }
        __syncwarp();
        fetch_hidden(g + G);  // into the slices the product above has just read: they are this warp's alone
        __syncthreads();

        // ---- this warp's tokens of the group ----
#pragma unroll 1
        for (int k = wt; k < TB; k += wstep) {
            const long long t = t_next;
            const bool valid = v_next, last = k + wstep >= TB;
            const unsigned char *row = row_next;
            t_next = next_token(g_next, k_next);
            id_next = t_next >= 0 ? id_of(t_next) : -1;
            // softmax numerators (Eq. 4): lane e <-> expert e; even slices and odd slices, then the two
            float z = 0.f;
            {
                const float *z_in = partial + k * nw * N + (lane % N);
                float ze = 0.f, zo = 0.f;
                for (int w = 0; w < nw; w += 2) {
                    ze += z_in[w * N];
                    if (w + 1 < nw) zo += z_in[(w + 1) * N];
                }
                z = ze + zo;
            }
            if (last && g + G < p.groups) named_bar_arrive(1, 2 * nw * 32);
            float shift = 0.f;  // the maximum, only where exp would leave the comfortable range
            if (__any_sync(0xffffffffu, !(fabsf(z) < 80.f))) shift = warp_max(z);
            const float e = expf(z - shift);
            if (lane < N) gates[lane] = e;
            __syncwarp();
            float es[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int j = 0; j < N; j += 4) {
                const float4 g4 = *reinterpret_cast<const float4 *>(gates + j);
                es[0] += g4.x, es[1] += g4.y, es[2] += g4.z, es[3] += g4.w;
            }
            const float esum = (es[0] + es[1]) + (es[2] + es[3]);
            const float inv = __frcp_rn(esum);
            if (p.gates_out && part == 0 && t >= 0 && lane < N) p.gates_out[t * N + lane] = e / esum;
            if (!valid && t >= 0 && part == 0 && lane == 0 && p.status) atomicOr(p.status, MOLE_STATUS_BAD_ID);

            v_next = id_next >= 0 && id_next < p.rows;
            row_next = static_cast<const unsigned char *>(p.lut) + static_cast<size_t>(v_next ? id_next : 0) * row_bytes + lane_off;
            const unsigned char *res_g = static_cast<const unsigned char *>(p.residual ? p.residual : p.hidden) + static_cast<size_t>(t < 0 ? 0 : t) * d * 2 + lane_off;
            unsigned char *out_g = static_cast<unsigned char *>(p.out) + static_cast<size_t>(t < 0 ? 0 : t) * d * 2 + lane_off;
#pragma unroll 1
            for (int pass = 0; pass < npass; ++pass) {
                const bool on = t >= 0 && pass * 256 + lane * 8 < cols;
                uint4 res = make_uint4(0u, 0u, 0u, 0u);
                if (on) res = ldcg_v4(res_g + pass * 512);
                float s[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) s[i] = 0.f;
                auto accumulate = [&](const uint4 (&r)[EB], int batch) {
#pragma unroll
                    for (int j = 0; j < EB; j += 4) {
                        const float4 g4 = *reinterpret_cast<const float4 *>(gates + batch * EB + j);
                        Elem<__nv_bfloat16>::fma_row(s, r[j], g4.x);
                        Elem<__nv_bfloat16>::fma_row(s, r[j + 1], g4.y);
                        Elem<__nv_bfloat16>::fma_row(s, r[j + 2], g4.z);
                        Elem<__nv_bfloat16>::fma_row(s, r[j + 3], g4.w);
                    }
                };
#pragma unroll
                for (int b = 0; b < BATCHES; b += 2) {
                    load(rb, row, pass, b + 1, valid);
                    accumulate(ra, b);
                    if (b + 2 < BATCHES) load(ra, row, pass, b + 2, valid);
                    else if (pass + 1 < npass) load(ra, row, pass + 1, 0, valid);
                    else load(ra, row_next, 0, 0, v_next);
                    accumulate(rb, b + 1);
                }
                if (valid) {
                    uint32_t rw[4] = {res.x, res.y, res.z, res.w};
#pragma unroll
                    for (int w = 0; w < 4; ++w) {
                        const __nv_bfloat162 v = __floats2bfloat162_rn(fmaf(s[2 * w], inv, __uint_as_float(rw[w] << 16)),
                                                                       fmaf(s[2 * w + 1], inv, __uint_as_float(rw[w] & 0xffff0000u)));
                        rw[w] = *reinterpret_cast<const uint32_t *>(&v);
                    }
                    res = make_uint4(rw[0], rw[1], rw[2], rw[3]);
                }
                if (on) *reinterpret_cast<uint4 *>(out_g + pass * 512) = res;
            }
            __syncwarp();  // the numerators have been read
        }
        if (wt >= TB && g + G < p.groups) named_bar_arrive(1, 2 * nw * 32);  // a warp without a token
    }
    cp_async_wait_all();
}

#endif  // __CUDACC__

}  // namespace mole
