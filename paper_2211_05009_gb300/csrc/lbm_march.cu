// lbm_march.cu -- launches of the fused kernel (lbm_march.cuh): up to kMarchSteps plain time steps of
// a single cavity in one pass over memory.
#include "lbm_internal.h"
#include "lbm_march.cuh"

namespace lbm {

namespace {
constexpr int kV = 4, kBY = 4;  // nodes per lane, warps per block
// Resident blocks per SM (4 warps each) the register budget is sized for, 168 registers (2048^2, us a step
// with 2 / 3 / 4 blocks: f32s 27.4 / 21.8 / 21.7, f32 36.0 / 30.9 / 44.4).
constexpr int kBlocks = 3;

template <typename S, bool SHIFTED, bool FULL>
cudaError_t launch_march_t(const MarchArgs& m, cudaStream_t st) {
    constexpr int smem = kBY * march_ring_bytes<S, kV, kMarchSteps>();
    auto* k = k_march<S, SHIFTED, kV, kMarchSteps, FULL, kBY, kBlocks>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    k<<<(m.g.warps() + kBY - 1) / kBY, dim3(32, kBY), smem, st>>>(m);
    return cudaGetLastError();
}

template <typename S, bool SHIFTED>
cudaError_t launch_march_s(const StepArgs& a, int steps, int sms, cudaStream_t st) {
    using G = StripGeometry<kV, kMarchSteps>;
    MarchArgs m;
    m.a = a;
    m.n = steps;
    // One wave: as many segments as the GPU holds warps, none shorter than two rows (a wall row and
    // its inner row stay together).
    m.g.strips = G::strips(a.nx);
    const int slots = sms * kBlocks * kBY;
    const int segs = slots / m.g.strips;
    m.g.segs = segs < 1 ? 1 : (segs > a.ny / 2 ? a.ny / 2 : segs);
    m.g.esegs = m.g.segs;
    if (steps == kMarchSteps) return launch_march_t<S, SHIFTED, true>(m, st);
    return launch_march_t<S, SHIFTED, false>(m, st);
}
}  // namespace

int march_columns(int nx) {
    using G = StripGeometry<kV, kMarchSteps>;
    return G::strips(nx) * G::kWidth;
}

cudaError_t launch_march(int dtype, const StepArgs& a, int steps, int sms, cudaStream_t st) {
    if (steps < 1 || steps > kMarchSteps) return cudaErrorInvalidValue;
    switch (dtype) {
        case 1: return launch_march_s<float, false>(a, steps, sms, st);
        case 2: return launch_march_s<float, true>(a, steps, sms, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace lbm
