// Host side of the tensor-core kernel (mole_mma.cuh): the shapes it covers, a launch's geometry, its tensor maps.
#include <string.h>

#include "mole_mma.cuh"

namespace mole {

constexpr int kSmemBlock = 227 * 1024, kSmemSM = 228 * 1024;

typedef void (*MmaKernel)(const CUtensorMap, const CUtensorMap, const MmaParams);
struct MmaVariant {
    MmaKernel fn;
    const char *name;
};
#define MOLE_MMA(N, CS) (norm ? MmaVariant{mole_mma_kernel<N, 1, CS>, "mma<" #N ",1," #CS ">"} : MmaVariant{mole_mma_kernel<N, 0, CS>, "mma<" #N ",0," #CS ">"})
static MmaVariant pick_mma(int N, int cs, bool norm)
{
    switch (N * 8 + cs) {
        case 8 * 8 + 1: return MOLE_MMA(8, 1);
        case 8 * 8 + 2: return MOLE_MMA(8, 2);
        case 16 * 8 + 1: return MOLE_MMA(16, 1);
        case 16 * 8 + 2: return MOLE_MMA(16, 2);
        case 32 * 8 + 1: return MOLE_MMA(32, 1);
        case 32 * 8 + 2: return MOLE_MMA(32, 2);
        case 32 * 8 + 4: return MOLE_MMA(32, 4);
        default: return MmaVariant{nullptr, "none"};
    }
}

static int smem_of(int N, int d, int cs, int ws, int rs, bool norm) { return static_cast<int>(mma_smem(N, d, cs, ws, rs, norm ? 1 : 0).total); }

// Blocks per token: as few as keep a block's part of a token's rows at 32 KB and its compute warps at eight; 0: not covered.
static int mma_blocks(int N, int d)
{
    for (int cs = 1; cs <= 4; cs *= 2) {
        if (d % (kMmaCols * cs) != 0) return 0;
        const int dl = d / cs;
        if (dl > 8 * kMmaCols || N * dl * 2 > 32 * 1024) continue;
        return pick_mma(N, cs, false).fn ? cs : 0;
    }
    return 0;
}

// Whether a fused step of M tokens runs here.  Up to one block per SM: every shape but d = 768 and 1024 with N = 16, which have
// kernels with the sizes compiled in (mole_slice.cuh: 10.5 against 17.6 us for 12 layers of 768, 64 tokens).  Up to two blocks per SM: where a block's part
// is small (N = 8, d = 1024, 250 tokens, 10 layers: 15.4 against 19.1 us; not N = 32, d = 512: 27.3 against 22.2) or the rows are so
// wide that the ring kernel cuts them finely (1B shape, 64 tokens: 36.5 against 53.2).  Beyond that a second wave starts where
// the ring kernel has the next token's rows in flight already.
bool mma_preferred(long long M, int dtype, int N, int d, int sms)
{
    if (dtype != MOLE_DTYPE_BF16 || (N != 8 && N != 16 && N != 32) || d % kMmaCols != 0 || d > kMmaMaxSlices * kMmaCols) return false;
    if (N == 16 && (d == 768 || d == 1024)) return false;
    const int cs = mma_blocks(N, d);
    if (!cs) return false;
    if (M * cs <= sms) return true;
    return M * cs <= 2LL * sms && (N * (d / cs) * 2 <= 24 * 1024 || N * d * 2 >= 128 * 1024);
}

int plan_mma(long long M, int N, int d, bool norm, int sms, bool prepare, MmaPlan *w)
{
    const int cs = mma_blocks(N, d);
    if (!cs) return MOLE_ERR_UNSUPPORTED_SHAPE;
    const MmaVariant v = pick_mma(N, cs, norm);
    w->fn = reinterpret_cast<const void *>(v.fn);
    w->name = v.name;
    w->cs = cs;
    w->threads = d / cs / 4 + 32;
    // one block per SM with deep rings, or two with shallower ones if that is what it takes to have all tokens resident
    // (clusters do not always fill the last SMs, so the driver is asked); fits: whether they are
    for (int want = 1; want <= 2; ++want) {
        const int budget = kSmemSM / want - 1024 < kSmemBlock ? kSmemSM / want - 1024 : kSmemBlock;
        int ws = 2, rs = kMmaMaxSlots;
        while (rs > 2 && smem_of(N, d, cs, ws, rs, norm) > budget) --rs;
        if (smem_of(N, d, cs, ws, rs, norm) > budget) ws = 1;
        if (smem_of(N, d, cs, ws, rs, norm) > budget) {
            if (want == 1) return MOLE_ERR_UNSUPPORTED_SHAPE;
            break;
        }
        w->w_slots = ws;
        w->r_slots = rs;
        w->smem = smem_of(N, d, cs, ws, rs, norm);
        long long resident = static_cast<long long>(want) * sms / cs;
        if (prepare) {
            int rc = ensure_smem_opt_in(w->fn, w->smem);
            if (rc != MOLE_OK) return rc;
            cudaLaunchConfig_t cfg;
            memset(&cfg, 0, sizeof cfg);
            cfg.gridDim = dim3(static_cast<unsigned>(cs), 1, 1);
            cfg.blockDim = dim3(static_cast<unsigned>(w->threads), 1, 1);
            cfg.dynamicSmemBytes = w->smem;
            int n = 0;
            if (cs > 1) {
                MOLE_CUDA_TRY(cudaOccupancyMaxActiveClusters(&n, w->fn, &cfg));
            } else {
                MOLE_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, v.fn, w->threads, w->smem));
                n *= sms;
            }
            resident = n > 0 ? n : 1;
        }
        w->fits = M <= resident;
        if (w->fits) break;
    }
    return MOLE_OK;
}

// Tensor maps of a launch: the router matrices [L][d N / 64][64] in boxes of a block's part, 128 bytes to a row, and the tables
// [L][rows][64-column chunk][expert][64] in boxes of one token's rows (a block's part of them).  A map depends on nothing but
// addresses and sizes; a decoding loop meets the same ones again and again, so each thread keeps its last few (encoding takes
// about as long as a launch).
struct MapKey {
    const void *base;
    long long stride, rows;
    int N, d, L, cs, what;
    bool operator==(const MapKey &o) const
    {
        return base == o.base && stride == o.stride && rows == o.rows && N == o.N && d == o.d && L == o.L && cs == o.cs && what == o.what;
    }
};
static bool encode_map(const MapKey &k, CUtensorMap *map)
{
    EncodeTiledFn enc = encode_tiled();
    if (!enc) return false;
    const cuuint32_t one[5] = {1, 1, 1, 1, 1};
    CUresult r;
    const cuuint64_t row = static_cast<cuuint64_t>(k.N) * k.d * 2;
    if (k.L > 1 && (k.stride < 16 || k.stride >= (1LL << 40) || (k.stride & 15))) return false;
    if (k.what == 0) {
        const int w_rows = k.d / k.cs * k.N / 64;  // at most 256: a block's part is 32 KB
        const cuuint64_t dims[3] = {64, static_cast<cuuint64_t>(k.d) * k.N / 64, static_cast<cuuint64_t>(k.L)};
        const cuuint64_t strides[2] = {128, k.L > 1 ? static_cast<cuuint64_t>(k.stride) : row};
        const cuuint32_t box[3] = {64, static_cast<cuuint32_t>(w_rows), 1};
        r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(k.base), dims, strides, box, one, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    } else {
        const cuuint64_t dims[5] = {64, static_cast<cuuint64_t>(k.N), static_cast<cuuint64_t>(k.d) / 64, static_cast<cuuint64_t>(k.rows), static_cast<cuuint64_t>(k.L)};
        const cuuint64_t strides[4] = {static_cast<cuuint64_t>(k.d) * 2, 128, row, k.L > 1 ? static_cast<cuuint64_t>(k.stride) : row};
        const cuuint32_t box[5] = {64, static_cast<cuuint32_t>(k.N), static_cast<cuuint32_t>(k.d / k.cs / 64), 1, 1};
        r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void *>(k.base), dims, strides, box, one, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    }
    return r == CUDA_SUCCESS;
}
static const CUtensorMap *map_for(const MapKey &k)
{
    constexpr int kEntries = 128;
    struct Entry {
        bool used = false;
        MapKey key;
        alignas(64) CUtensorMap map;
    };
    thread_local Entry cache[kEntries];
    const uint64_t h = (reinterpret_cast<uintptr_t>(k.base) >> 4) * 0x9E3779B97F4A7C15ull + static_cast<uint64_t>(k.what) * 0x5851F42D4C957F2Dull;
    Entry &e = cache[h >> 57];
    if (e.used && e.key == k) return &e.map;
    e.used = false;
    if (!encode_map(k, &e.map)) return nullptr;
    e.key = k;
    e.used = true;
    return &e.map;
}

// (a fused step has neither gates to write nor a residual of its own)
int launch_mma(const StepLaunch &a, const MmaPlan &w, uint32_t wait_polls, bool *taken)
{
    *taken = false;
    CUtensorMap w_map, r_map;
    const CUtensorMap *m = map_for({a.w_router, a.wr_stride, 0, a.N, a.d, a.L, w.cs, 0});
    if (!m) return MOLE_OK;
    w_map = *m;
    m = map_for({a.lut, a.lut_stride, a.rows, a.N, a.d, a.L, w.cs, 1});
    if (!m) return MOLE_OK;
    r_map = *m;
    *taken = true;
    MmaParams p;
    p.hidden = a.hidden;
    p.row_index = a.row_index;
    p.norm_weight = a.norm_weight;
    p.out = a.out;
    p.status = a.status;
    p.norm_stride = a.norm_stride;
    p.rows = a.rows;
    p.d = a.d;
    p.L = a.L;
    p.w_slots = w.w_slots;
    p.r_slots = w.r_slots;
    p.norm_eps = a.norm_eps;
    p.inv_d = 1.0f / static_cast<float>(a.d);
    p.flags = a.flags;
    p.wait_polls = wait_polls;
    void *args[3] = {&w_map, &r_map, &p};
    return launch_pdl(w.fn, static_cast<unsigned>(a.M * w.cs), static_cast<unsigned>(w.threads), w.smem, a.stream, args, (a.flags & MOLE_FLAG_CHAIN) != 0);
}

}  // namespace mole
