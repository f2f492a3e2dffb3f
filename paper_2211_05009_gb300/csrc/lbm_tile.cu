// lbm_tile.cu -- launches of the shared-memory tile kernel (lbm_tile.cuh): several plain time steps of
// a small cavity per launch.
#include <atomic>

#include "lbm_internal.h"
#include "lbm_tile.cuh"

namespace lbm {

namespace {
constexpr int kTileSteps = 4, kTileLow = 10, kTileHigh = 24;  // steps of a launch, rows a tile owns
constexpr int tile_bytes(int oh, int n, int elem) { return 2 * 9 * kTileCols * (oh + 2 * n) * elem; }

// Opt in to the largest tile's shared memory, once per device.  The attribute belongs to the kernel on the
// device: a launch that set it to its own size would lower it between another context's set and launch
// (contexts are independent, each with a thread of its own), and that launch would be refused.
template <typename S, bool SHIFTED>
cudaError_t opt_in() {
    static std::atomic<unsigned long long> done{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
    if (done.load(std::memory_order_relaxed) & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(k_tile<S, SHIFTED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             tile_bytes(kTileHigh, kTileSteps, (int)sizeof(S)));
    if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_relaxed);
    return e;
}

template <typename S, bool SHIFTED>
cudaError_t launch_tile_t(const StepArgs& a, const TilePlan& p, int n, cudaStream_t st) {
    const int smem = tile_bytes(p.oh, n, (int)sizeof(S));
    const cudaError_t e = opt_in<S, SHIFTED>();
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
    p.steps = kTileSteps;
    p.ow = kTileCols - 2 * p.steps;
    // Rows so that the row pairs of a step fill the warps once (10 + 2 x 3 rows, 8 pairs) or twice
    // (24): the taller tile computes fewer nodes twice, the lower one makes more blocks.  The lower one
    // up to two blocks for each of the 152 SMs (us a step, low / high: f32s 96^2 1.1 / 1.5, 192x380 with 304 low
    // blocks 1.37 / 1.60, 288x255 with 312 1.50 / 1.61; q16s 1.6 / 2.5, 2.36 / 2.58, 2.71 / 2.58).
    const int cols = (nx + p.ow - 1) / p.ow;
    p.oh = (long long)cols * ((ny + 9) / 10) <= 2 * 152 ? kTileLow : kTileHigh;
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
