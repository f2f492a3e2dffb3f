// lbm_tile.cu -- launches of the shared-memory tile kernel (lbm_tile.cuh): several plain time steps of
// a small cavity per launch.
#include "lbm_internal.h"
#include "lbm_tile.cuh"

namespace lbm {

namespace {
template <typename S, bool SHIFTED>
cudaError_t launch_tile_t(const StepArgs& a, const TilePlan& p, int n, cudaStream_t st) {
    const int smem = 2 * 9 * kTileCols * (p.oh + 2 * n) * (int)sizeof(S);
    const cudaError_t e = cudaFuncSetAttribute(k_tile<S, SHIFTED>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    TileArgs m;
    m.a = a;
    m.p = p;
    m.n = n;
    const dim3 grid((unsigned)((a.nx + p.shift_x + p.ow - 1) / p.ow), (unsigned)((a.ny + p.shift_y + p.oh - 1) / p.oh));
    k_tile<S, SHIFTED><<<grid, 32 * kTileWarps, smem, st>>>(m);
    return cudaGetLastError();
}
}  // namespace

TilePlan tile_plan(int nx, int ny) {
    TilePlan p{};
    p.steps = 4;
    p.ow = kTileCols - 2 * p.steps;
    // Rows so that the row pairs of a step fill the warps once (10 + 2 x 3 rows, 8 pairs) or twice
    // (24): the taller tile computes fewer nodes twice, the lower one makes more blocks.
    const int cols = (nx + p.ow - 1) / p.ow;
    p.oh = (long long)cols * ((ny + 9) / 10) <= 2 * 148 ? 10 : 24;
    // a wall is never the only column or row of a tile; columns move by a copy's alignment
    p.shift_x = nx % p.ow == 1 ? 4 : 0;
    p.shift_y = ny % p.oh == 1 ? 1 : 0;
    return p;
}

cudaError_t launch_tile(int dtype, const StepArgs& a, const TilePlan& p, int steps, cudaStream_t st) {
    if (steps < 1 || steps > p.steps) return cudaErrorInvalidValue;
    switch (dtype) {
        case 1: return launch_tile_t<float, false>(a, p, steps, st);
        case 2: return launch_tile_t<float, true>(a, p, steps, st);
        case 3: return launch_tile_t<__half, true>(a, p, steps, st);
        case 4: return launch_tile_t<__nv_bfloat16, true>(a, p, steps, st);
        case 5: return launch_tile_t<q16, true>(a, p, steps, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace lbm
