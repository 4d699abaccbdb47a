// Host side of the tensor-core kernel (mole_mma.cuh): the shapes it covers, a launch's geometry, its tensor maps.
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include "mole_mma.cuh"

namespace mole {

constexpr int kSmemBlock = 227 * 1024, kSmemSM = 228 * 1024;

typedef void (*MmaKernel)(const CUtensorMap, const CUtensorMap, const MmaParams);

template <int N, int CS>
static MmaKernel pick_mma_tb(int tb, bool norm)
{
    if (tb == 1) return norm ? mole_mma_kernel<N, 1, 1, CS> : mole_mma_kernel<N, 1, 0, CS>;
    return norm ? mole_mma_kernel<N, 8, 1, CS> : mole_mma_kernel<N, 8, 0, CS>;
}
static MmaKernel pick_mma(int N, int cs, int tb, bool norm)
{
    switch (N * 8 + cs) {
        case 8 * 8 + 1: return pick_mma_tb<8, 1>(tb, norm);
        case 8 * 8 + 2: return pick_mma_tb<8, 2>(tb, norm);
        case 16 * 8 + 1: return pick_mma_tb<16, 1>(tb, norm);
        case 16 * 8 + 2: return pick_mma_tb<16, 2>(tb, norm);
        case 32 * 8 + 1: return pick_mma_tb<32, 1>(tb, norm);
        case 32 * 8 + 2: return pick_mma_tb<32, 2>(tb, norm);
        case 32 * 8 + 4: return pick_mma_tb<32, 4>(tb, norm);
        default: return nullptr;
    }
}

static int smem_of(int N, int d, int cs, int tb, int ws, int rs, bool norm) { return static_cast<int>(mma_smem(N, d, cs, tb, ws, rs, norm ? 1 : 0).total); }

// Blocks per token: as few as keep a block's part of a token's rows at 32 KB and its compute warps at eight; 0: not covered.
static int mma_blocks(int N, int d)
{
    for (int cs = 1; cs <= 4; cs *= 2) {
        if (d % (kMmaCols * cs) != 0) return 0;
        const int dl = d / cs;
        if (dl > 8 * kMmaCols || N * dl * 2 > 32 * 1024) continue;
        return pick_mma(N, cs, 1, false) ? cs : 0;
    }
    return 0;
}

bool mma_shape_ok(int dtype, int N, int d)
{
    return dtype == MOLE_DTYPE_BF16 && (N == 8 || N == 16 || N == 32) && d % kMmaCols == 0 && d <= 2048 && mma_blocks(N, d) > 0;
}

int plan_mma(long long M, int L, int N, int d, bool norm, int sms, bool prepare, MmaPlan *w)
{
    const int cs = mma_blocks(N, d);
    if (!cs) return MOLE_ERR_UNSUPPORTED_SHAPE;
    const long long per_sm_tokens = (M * cs + sms - 1) / sms;
    int tb = per_sm_tokens > 4 ? 8 : 1;
    if (const char *e = getenv("WTB")) tb = atoi(e);
    const long long groups = (M + tb - 1) / tb;
    if (groups > 0x1fffffff) return MOLE_ERR_TOO_LARGE;
    // blocks per SM aimed at
    const long long per_sm_blocks = (groups * cs + sms - 1) / sms;
    int want = static_cast<int>(per_sm_blocks < 1 ? 1 : (per_sm_blocks > (tb == 1 ? 4 : 2) ? (tb == 1 ? 4 : 2) : per_sm_blocks));
    if (const char *e = getenv("WBPS")) want = atoi(e);
    int ws = L > 1 ? 2 : 1, rs = 0;
    for (; want >= 1 && rs == 0; --want) {
        const int budget = kSmemSM / want - 1024 < kSmemBlock ? kSmemSM / want - 1024 : kSmemBlock;
        for (ws = L > 1 ? 2 : 1; ws >= 1 && rs == 0; --ws)
            for (int r = L > 1 || tb > 1 ? kMmaMaxSlots : 2; r >= (L > 1 ? 2 : 1); --r)
                if (smem_of(N, d, cs, tb, ws, r, norm) <= budget) {
                    rs = r;
                    break;
                }
        ++ws;
    }
    if (rs == 0) return MOLE_ERR_UNSUPPORTED_SHAPE;
    if (const char *e = getenv("WRS")) rs = atoi(e);
    if (const char *e = getenv("WWS")) ws = L > 1 ? atoi(e) : 1;
    w->w_slots = ws;
    w->r_slots = rs;
    w->smem = smem_of(N, d, cs, tb, ws, rs, norm);
    if (w->smem > kSmemBlock) return MOLE_ERR_UNSUPPORTED_SHAPE;
    const MmaKernel fn = pick_mma(N, cs, tb, norm);
    w->fn = reinterpret_cast<const void *>(fn);
    w->cs = cs;
    w->tb = tb;
    w->threads = d / cs / 4 + 32;
    w->groups = static_cast<int>(groups);
    int per_sm = 1;
    if (prepare) {
        int rc = ensure_smem_opt_in(w->fn, w->smem);
        if (rc != MOLE_OK) return rc;
        MOLE_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, w->threads, w->smem));
        if (per_sm < 1) per_sm = 1;
    }
    const long long resident = static_cast<long long>(per_sm) * sms / cs;
    w->grid = static_cast<int>(groups < resident ? groups : resident) * cs;
    if (getenv("WDBG")) fprintf(stderr, "mma M %lld L %d N %d d %d: cs %d tb %d ws %d rs %d smem %d per_sm %d grid %d\n", M, L, N, d, cs, tb, ws, rs, w->smem, per_sm, w->grid);
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
        const int w_rows = k.d / k.cs * k.N / 64;
        const cuuint64_t dims[3] = {64, static_cast<cuuint64_t>(k.d) * k.N / 64, static_cast<cuuint64_t>(k.L)};
        const cuuint64_t strides[2] = {128, k.L > 1 ? static_cast<cuuint64_t>(k.stride) : row};
        const cuuint32_t box[3] = {64, static_cast<cuuint32_t>(w_rows <= 256 ? w_rows : w_rows / 2), 1};
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
    p.residual = a.residual;
    p.row_index = a.row_index;
    p.norm_weight = a.norm_weight;
    p.out = a.out;
    p.gates_out = a.gates_out;
    p.status = a.status;
    p.norm_stride = a.norm_stride;
    p.M = a.M;
    p.rows = a.rows;
    p.d = a.d;
    p.L = a.L;
    p.groups = w.groups;
    p.w_slots = w.w_slots;
    p.r_slots = w.r_slots;
    p.norm_eps = a.norm_eps;
    p.flags = a.flags;
    p.wait_polls = wait_polls;
    void *args[3] = {&w_map, &r_map, &p};
    return launch_pdl(w.fn, static_cast<unsigned>(w.grid), static_cast<unsigned>(w.threads), w.smem, a.stream, args, (a.flags & MOLE_FLAG_CHAIN) != 0);
}

}  // namespace mole
