// Shared device helpers and host-side error plumbing of the MoLE sm_100a library.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "mole.h"

namespace mole {

// ---- host side -----------------------------------------------------------------------------
void set_cuda_error(cudaError_t e);  // remembers the text for mole_last_cuda_error()

#define MOLE_CUDA_TRY(expr)                       \
    do {                                          \
        cudaError_t e__ = (expr);                 \
        if (e__ != cudaSuccess) {                 \
            ::mole::set_cuda_error(e__);          \
            return MOLE_ERR_CUDA;                 \
        }                                         \
    } while (0)

inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
inline int elem_bytes(int dtype) { return dtype == MOLE_DTYPE_BF16 ? 2 : 4; }

// Launch description of the fused kernel (filled by plan_step, pure host arithmetic).
// A block owns whole tokens; it walks over its tokens and, for every token, over the L layers,
// pulling the router matrix (when it streams) and the table rows of each (token, layer) item, cut
// into d_split chunks, through a ring of `stages` shared-memory slots.
struct StepPlan {
    int d_split;        // chunks per item (of the router matrix, and of the rows)
    int dc;             // columns per router chunk (and per rows chunk when the rows are cut by columns)
    int consumers;      // threads that compute (a multiple of 32); one more warp issues the copies
    int threads;        // consumers + 32
    int stages;         // ring depth, in chunks
    int hring;          // hidden states of tokens in flight
    int slot_bytes;     // one ring slot
    int wr_in_ring;     // 1: the router chunks travel through the ring; 0: router matrix loaded once per block
    int smem;           // dynamic shared memory, bytes
    int blocks_per_sm;  // resident blocks per SM the shared memory allows
    int n_fast;         // N if the unrolled router path exists for it, else 0
    int rows_by_expert; // several chunks per item: 1 = the rows are cut by experts, 0 = by columns
    int lanes;          // combine: lanes per 16-byte column group (by columns) or column groups per lane (by experts)
};
// `by_columns`: never cut the rows by experts (kernel variants that exist for the column cut only)
// `sms`: SM count the plan is laid out for (< 1: the nominal 148 of a B200); `norm`: room for RMSNorm(hidden)
int plan_step(long long M, int L, int N, int d, int dtype, int d_split, StepPlan *plan, bool by_columns = false, int sms = 0,
              bool norm = false);

// One launch of the fused kernel over L chained layers (L == 1: a single layer).
// `row_index` is ids (resident mode) or slot (offload mode); `rows` the number of table rows
// that may be addressed.
struct StepLaunch {
    const void *hidden, *residual, *row_index, *lut, *w_router;
    void *out;
    float *gates_out;
    uint32_t *status;
    long long lut_stride, wr_stride;  // bytes between consecutive layers
    long long M;
    int L, N, d;
    long long rows;
    int dtype;
    uint32_t flags;
    int d_split;
    cudaStream_t stream;
    const void *norm_weight = nullptr;  // [d], dtype: the router reads RMSNorm(hidden); NULL: hidden itself
    long long norm_stride = 0;          // bytes between the scale vectors of consecutive layers
    float norm_eps = 0.f;
    int kernel = 0;  // MOLE_KERNEL_*: which kernel family runs the launch (0: the library's choice)
    bool first = false;  // the first of a step's chained layers
};
int launch_step(const StepLaunch &a);

// The prefill kernel (mole_tile.cu): the shapes it covers, one launch's geometry.
struct TilePlan {
    const void *fn;
    const char *name;
    int tb, threads, smem, groups, grid;
};
bool tile_shape_ok(int dtype, int N, int d);
int plan_tile(long long M, int N, int d, bool norm, int sms, bool prepare, TilePlan *t);
int launch_tile(const StepLaunch &a, const TilePlan &t);

// The tensor-core step kernel (mole_mma.cu): whether a fused step runs on it, one launch's geometry.  launch_mma leaves `taken`
// false, and launches nothing, where the tables' strides do not make tensor maps.
struct MmaPlan {
    const void *fn;
    const char *name;
    int cs, threads, smem, w_slots, r_slots;
    bool fits;  // all blocks are resident at once
};
bool mma_preferred(long long M, int dtype, int N, int d, int sms);
int plan_mma(long long M, int N, int d, bool norm, int sms, bool prepare, MmaPlan *w);
int launch_mma(const StepLaunch &a, const MmaPlan &w, uint32_t wait_polls, bool *taken);

// cuTensorMapEncodeTiled, looked up once (mole_builder.cu); nullptr if the driver has none
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled();

// Every layer kernel is launched with programmatic stream serialization: its blocks may be set up while the kernel before it
// on the stream still runs, and it waits for that kernel itself -- first thing (pdl_enter), or, with MOLE_FLAG_CHAIN, before
// it reads the hidden state.  Back-to-back launches of one token of a 160M-shaped layer: 4.9 -> 3.4 us.
// (Not inside a stream capture unless chained: there the attribute costs a graph of one kernel 2 us.  `alone`: not at all.)
int launch_pdl(const void *fn, unsigned grid, unsigned threads, int smem, cudaStream_t stream, void **args, bool chained, bool alone = false);

// kernels that need more than 48 KB of dynamic shared memory opt in once per device
int ensure_smem_opt_in(const void *fn, int smem);
int sm_count(int *out, int *dev_out = nullptr);  // SM count of the current device, asked once per device
// resident blocks per SM of a launch, asked once per (kernel, threads, shared memory) and thread
int blocks_per_sm(const void *fn, int threads, int smem, int *out);
// poll limit of the bounded device-side waits (the default unless a debugging variable shortens it)
uint32_t current_wait_polls();
// MOLE_FORCE_BUILDER_TILES: 1 single blocks, 2 pairs; otherwise the builder chooses
int forced_builder_tiles();

// the fused layer over a quantised table (mole_quant.cu): single layer, bf16 activations
bool quant_layer_shape_ok(int N, int d, int format, int block);
int launch_quant_layer(const StepLaunch &a, int format, int block, uint32_t wait_polls);
// ... and the fused step over L quantised tables, the same bits as L single layers
bool quant_step_preferred(long long M, int N, int d, int format, int block, int sms);
// name and launch shape of the kernel that runs M tokens and L layers over quantised tables (L > 1: MOLE_STEP_AUTO's choice)
struct QuantVariant {
    const char *name;
    int threads, smem;
};
QuantVariant quant_variant(long long M, int L, int N, int d, int format, int block, bool norm, int sms);
int launch_quant_step(const StepLaunch &a, int format, int block, uint32_t wait_polls);

#ifdef __CUDACC__
// ---- device side ---------------------------------------------------------------------------

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// mbarrier + bulk-copy (TMA, untiled, each copy into this block's own shared memory only) primitives
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Global -> this block's shared memory; both addresses 16-byte aligned, bytes a multiple of 16.
__device__ __forceinline__ void bulk_g2s(void *dst_smem, const void *src_gmem, uint32_t bytes, uint64_t *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst_smem)),
                 "l"(src_gmem), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// Ask L2 for a span of global memory (no destination, no completion to wait for); address 16-byte aligned,
// bytes a multiple of 16.
__device__ __forceinline__ void bulk_prefetch_l2(const void *src_gmem, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src_gmem), "r"(bytes) : "memory");
}

// Bounded wait on a bulk-copy barrier.  Returns false if the data never arrived.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity, uint32_t max_polls)
{
    for (uint32_t i = 0; i < max_polls; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if (i > 64) __nanosleep(64);
    }
    return false;
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Barrier over a subset of the block's warps (id 1..15, count a multiple of 32).
__device__ __forceinline__ void named_bar_sync(int id, int count)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}
// Count this warp in at a named barrier without waiting for it.
__device__ __forceinline__ void named_bar_arrive(int id, int count)
{
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_proxy_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }

// programmatic dependent launch
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Loads of the norm's scale, behind pdl_wait(): the kernel before a chained launch may have written it, so that the read-only path
// (__ldg, which may also be moved ahead of the wait) is closed; but every block reads the same few lines, so that they are to come from L1
// where they can (past it, 12 layers of 16 x 768 NF4, 400 tokens: 63.4 -> 86.0 us).
__device__ __forceinline__ uint32_t ld_scale_u16(const void *p)
{
    uint32_t v;
    asm volatile("ld.global.u16 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint2 ld_scale_v2(const void *p)
{
    uint2 v;
    asm volatile("ld.global.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint4 ld_scale_v4(const void *p)
{
    uint4 v;
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
// Top of a kernel launched by launch_pdl.  Unless the caller vouched that the kernel before this one writes neither ids nor
// tables nor routers (MOLE_FLAG_CHAIN), it waits for that kernel before anything is read -- and before the next launch may
// start: that one may be chained and would otherwise read tables while their writer, two launches back, still runs.
__device__ __forceinline__ void pdl_enter(uint32_t flags)
{
    if (!(flags & MOLE_FLAG_CHAIN)) {
        pdl_wait();
        fence_proxy_async_global();
    }
    pdl_launch_dependents();
}

// Explicit shared-space accesses (32-bit shared addresses): the hot loops index slots of the
// ring through run-time offsets, and these keep every access on the shared-memory path.
__device__ __forceinline__ uint4 lds128(uint32_t a)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ uint2 lds64(uint32_t a)
{
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}
__device__ __forceinline__ uint32_t lds32(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ uint32_t lds16(uint32_t a)
{
    unsigned short v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts128(uint32_t a, const uint4 &v)
{
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void sts64(uint32_t a, const uint2 &v)
{
    asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(v.x), "r"(v.y) : "memory");
}
__device__ __forceinline__ void sts32(uint32_t a, uint32_t v)
{
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// Warp-wide matrix loads and products, 16-byte asynchronous copies.
__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm_x4_trans(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
// c += a b: A 16 x 16, B 16 x 8, bf16 products, fp32 sums
__device__ __forceinline__ void mma16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// ... A 16 x 8, B 8 x 8
__device__ __forceinline__ void mma8(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t b0)
{
    asm("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5}, {%6}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(b0));
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }
// RMSNorm's factor, 1 / sqrt(mean + eps), by the correctly rounded root and division: 0 where the sum of squares overflows
__device__ __forceinline__ float rms_scale(float total, int d, float eps) { return 1.0f / sqrtf(total / static_cast<float>(d) + eps); }

// 16-byte vectors of the two storage types
template <typename T>
struct Elem;
template <>
struct Elem<__nv_bfloat16> {
    static constexpr int VEC = 8;
    static __device__ __forceinline__ void unpack(const uint4 &v, float (&f)[8])
    {
        f[0] = __uint_as_float(v.x << 16);
        f[1] = __uint_as_float(v.x & 0xffff0000u);
        f[2] = __uint_as_float(v.y << 16);
        f[3] = __uint_as_float(v.y & 0xffff0000u);
        f[4] = __uint_as_float(v.z << 16);
        f[5] = __uint_as_float(v.z & 0xffff0000u);
        f[6] = __uint_as_float(v.w << 16);
        f[7] = __uint_as_float(v.w & 0xffff0000u);
    }
    // acc[0..7] += g * (the 8 values of v): the weighted sum's inner step.  Two values per instruction on the
    // packed fp32 pipe (fma.rn.f32x2: two independent IEEE fmas, the same bits as eight fmaf).
    static __device__ __forceinline__ void fma_row(float (&acc)[8], const uint4 &v, float g)
    {
        const float2 g2 = make_float2(g, g);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float2 r = __ffma2_rn(g2, make_float2(__uint_as_float(w[k] << 16), __uint_as_float(w[k] & 0xffff0000u)),
                                        make_float2(acc[2 * k], acc[2 * k + 1]));
            acc[2 * k] = r.x;
            acc[2 * k + 1] = r.y;
        }
    }
    // element i of an array in shared memory (32-bit shared address)
    static __device__ __forceinline__ float lds_scalar(uint32_t base, int i) { return __uint_as_float(lds16(base + 2 * i) << 16); }
    // the same element as a raw 16-bit operand of the mixed-precision fma below
    typedef unsigned short H;
    static __device__ __forceinline__ H lds_h(uint32_t base, int i)
    {
        unsigned short v;
        asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(base + 2u * i));
        return v;
    }
    // acc[e] += v[e] * h for the 8 values of a vector, through sm_100's mixed-precision fma
    // (fma.rn.f32.bf16: bf16 x bf16 products are exact in fp32, one rounding at the add -- the
    // same result as widening both operands and calling fmaf, without the widening instructions)
    static __device__ __forceinline__ void fma_elem(float &acc, const uint4 &v, int e, H h)
    {
        const uint32_t w = e < 2 ? v.x : (e < 4 ? v.y : (e < 6 ? v.z : v.w));
        unsigned short lo, hi;
        asm("mov.b32 {%0, %1}, %2;" : "=h"(lo), "=h"(hi) : "r"(w));
        asm("fma.rn.f32.bf16 %0, %1, %2, %0;" : "+f"(acc) : "h"((e & 1) ? hi : lo), "h"(h));
    }
};
template <>
struct Elem<float> {
    static constexpr int VEC = 4;
    static __device__ __forceinline__ void unpack(const uint4 &v, float (&f)[4])
    {
        f[0] = __uint_as_float(v.x);
        f[1] = __uint_as_float(v.y);
        f[2] = __uint_as_float(v.z);
        f[3] = __uint_as_float(v.w);
    }
    static __device__ __forceinline__ void fma_row(float (&acc)[4], const uint4 &v, float g)
    {
        acc[0] = fmaf(g, __uint_as_float(v.x), acc[0]);
        acc[1] = fmaf(g, __uint_as_float(v.y), acc[1]);
        acc[2] = fmaf(g, __uint_as_float(v.z), acc[2]);
        acc[3] = fmaf(g, __uint_as_float(v.w), acc[3]);
    }
    static __device__ __forceinline__ float lds_scalar(uint32_t base, int i) { return __uint_as_float(lds32(base + 4 * i)); }
    typedef float H;
    static __device__ __forceinline__ H lds_h(uint32_t base, int i) { return __uint_as_float(lds32(base + 4 * i)); }
    static __device__ __forceinline__ void fma_elem(float &acc, const uint4 &v, int e, H h)
    {
        const uint32_t w = e == 0 ? v.x : (e == 1 ? v.y : (e == 2 ? v.z : v.w));
        acc = fmaf(h, __uint_as_float(w), acc);
    }
};
#endif  // __CUDACC__

}  // namespace mole
