// Host side of the prefill kernel (mole_tile.cuh): the shapes it covers and a launch's geometry.
#include <string.h>

#include "mole_tile.cuh"

namespace mole {

constexpr int kSmemBlock = 227 * 1024;

typedef void (*TileKernel)(const TileParams);

template <int N, int D>
static TileKernel pick_tile_p(bool norm, int parts)
{
    switch (parts) {
        case 1: return norm ? mole_tile_kernel<N, 1, D, 1> : mole_tile_kernel<N, 0, D, 1>;
        case 2: return norm ? mole_tile_kernel<N, 1, D, 2> : mole_tile_kernel<N, 0, D, 2>;
        default: return nullptr;
    }
}
template <int N>
static TileKernel pick_tile_wide(bool norm, int parts)
{
    if (parts == 2) return norm ? mole_tile_kernel<N, 1, 2048, 2> : mole_tile_kernel<N, 0, 2048, 2>;
    return norm ? mole_tile_kernel<N, 1, 2048, 4> : mole_tile_kernel<N, 0, 2048, 4>;
}
static TileKernel pick_tile(int N, bool norm, int d, int parts)
{
    if (N == 16 && d == 768) return pick_tile_p<16, 768>(norm, parts);
    if (N == 16 && d == 1024) return pick_tile_p<16, 1024>(norm, parts);
    if (N == 32 && d == 1024) return pick_tile_p<32, 1024>(norm, parts);
    if (N == 16 && d == 2048) return pick_tile_wide<16>(norm, parts);
    if (N == 32 && d == 2048) return pick_tile_wide<32>(norm, parts);
    if (d <= 1024) {
        switch (N) {
            case 8: return pick_tile_p<8, kTileNarrow>(norm, parts);
            case 16: return pick_tile_p<16, kTileNarrow>(norm, parts);
            case 32: return pick_tile_p<32, kTileNarrow>(norm, parts);
        }
    } else {
        switch (N) {
            case 8: return pick_tile_p<8, kTileWide>(norm, parts);
            case 16: return pick_tile_p<16, kTileWide>(norm, parts);
            case 32: return pick_tile_p<32, kTileWide>(norm, parts);
        }
    }
    return nullptr;
}

bool tile_shape_ok(int dtype, int N, int d)
{
    return dtype == MOLE_DTYPE_BF16 && (N == 8 || N == 16 || N == 32) && d % kSliceCols == 0 && d <= kSliceCols * kTileMaxWarps;
}

int plan_tile(long long M, int N, int d, bool norm, int sms, bool prepare, TilePlan *t)
{
    const int warps = d / kSliceCols;
    // Groups of about eight tokens, a warp per token, or two warps per token where there are more warps than that; several tokens
    // per warp where there are fewer.  A launch whose smaller groups -- one token per warp, then twice the warps per token -- are
    // still all resident at once takes those: more blocks with less to do one after the other (410M shape, 1 300 tokens: 12.4
    // -> 10.3 us; beyond one wave the larger groups win, 16 384 tokens: 54 against 58 us).
    int parts = warps > 8 && warps % 2 == 0 ? 2 : 1;
    int tb = warps >= 8 ? warps / parts : warps * (8 / warps);
    for (int step = 0; step < 3; ++step) {
        if (step == 1) {
            if (tb <= warps / parts) continue;
            tb = warps / parts;
        } else if (step == 2) {
            if (warps % (2 * parts) != 0 || (parts == 2 && !(d == 2048 && N >= 16))) break;
            parts *= 2;
            tb = warps / parts;
        }
        while (tb > 1 && tile_smem(N, d, tb, norm ? 1 : 0).total > static_cast<uint32_t>(kSmemBlock)) --tb;
        const int smem = static_cast<int>(tile_smem(N, d, tb, norm ? 1 : 0).total);
        if (smem > kSmemBlock) return MOLE_ERR_UNSUPPORTED_SHAPE;
        const TileKernel fn = pick_tile(N, norm, d, parts);
        int per_sm = 1;
        if (prepare) {
            int rc = ensure_smem_opt_in(reinterpret_cast<void *>(fn), smem);
            if (rc != MOLE_OK) return rc;
            MOLE_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, d / 4, smem));
            if (per_sm < 1) per_sm = 1;
        }
        const long long groups = (M + tb - 1) / tb, resident = static_cast<long long>(per_sm) * sms;
        if (groups > 0x3fffffff) return MOLE_ERR_TOO_LARGE;
        if (step > 0 && groups > resident) break;
        t->fn = reinterpret_cast<void *>(fn);
        t->tb = tb;
        t->threads = d / 4;
        t->smem = smem;
        t->groups = static_cast<int>(groups);
        t->grid = static_cast<int>(groups < resident ? groups : resident);
    }
    return MOLE_OK;
}

int launch_tile(const StepLaunch &a, const TilePlan &t)
{
    TileParams p;
    p.hidden = a.hidden;
    p.residual = a.residual;
    p.row_index = a.row_index;
    p.lut = a.lut;
    p.w_router = a.w_router;
    p.norm_weight = a.norm_weight;
    p.out = a.out;
    p.gates_out = a.gates_out;
    p.status = a.status;
    p.M = a.M;
    p.rows = a.rows;
    p.d = a.d;
    p.tb = t.tb;
    p.groups = t.groups;
    p.norm_eps = a.norm_eps;
    p.flags = a.flags;
    void *args[1] = {&p};
    return launch_pdl(t.fn, static_cast<unsigned>(t.grid), static_cast<unsigned>(t.threads), t.smem, a.stream, args, (a.flags & MOLE_FLAG_CHAIN) != 0);
}

}  // namespace mole
