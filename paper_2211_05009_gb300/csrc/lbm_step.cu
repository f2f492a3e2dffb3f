// lbm_step.cu -- dispatch of the fused step kernel over storage types and launch shapes, and
// the fixed-order FP64 reduction that closes each 100-step checkpoint (Eq. 6 residual, mass).
#include <cmath>

#include "lbm_device.cuh"
#include "lbm_internal.h"

namespace lbm {

cudaError_t launch_step_f64(int cfg, const StepArgs& a, bool reduce, cudaStream_t st);
cudaError_t launch_step_f32(int cfg, const StepArgs& a, bool reduce, cudaStream_t st);
cudaError_t launch_step_f32s(int cfg, const StepArgs& a, bool reduce, cudaStream_t st);
cudaError_t launch_step_f16s(int cfg, const StepArgs& a, bool reduce, cudaStream_t st);
cudaError_t launch_step_bf16s(int cfg, const StepArgs& a, bool reduce, cudaStream_t st);
cudaError_t launch_step_q16s(int cfg, const StepArgs& a, bool reduce, cudaStream_t st);

namespace {
struct Shape {
    int V, R, BY;
};
// must match launch_step_cfg in lbm_step_kernel.cuh: FP64, FP32 storage, 16-bit storage
constexpr Shape kShapes[3][kRowConfigs] = {{{1, 2, 2}, {1, 2, 4}, {1, 1, 4}, {1, 4, 1}, {1, 2, 1}, {1, 1, 1}},
                                           {{2, 2, 2}, {2, 1, 4}, {1, 1, 4}, {2, 4, 1}, {2, 2, 4}, {2, 2, 2}},
                                           {{4, 2, 2}, {4, 1, 4}, {4, 2, 2}, {4, 4, 1}, {4, 2, 4}, {4, 4, 2}}};
}  // namespace

double q16_scale(int j, double U) {
    const double w = j == 0 ? 4.0 / 9.0 : (j < 5 ? 1.0 / 9.0 : 1.0 / 36.0);
    const double K = j == 0 ? 2.0 : (j < 5 ? 5.0 : 5.5);
    const double u = fabs(U) > 0.01 ? fabs(U) : 0.01;
    return 0.5 * exp2(ceil(log2(K * w * u)));  // 2 S_j = the power of two at or above K w u
}

QCodec q16_codec(double U) {
    QCodec q{};
    for (int j = 0; j < 9; ++j) {
        const double S = q16_scale(j, U);
        q.dec[j] = (float)(exp2(124.0) * S);
        q.enc[j] = (float)(exp2(-124.0) / S);
    }
    return q;
}

int default_step_config(int dtype, int nx, int ny) {
    const long long n = (long long)nx * ny;
    // FP64: one node per lane and one row per one-warp block at every size.  The FP64 pipe is the bound,
    // a warp's node takes 1.7 us of it by itself, and the smaller the piece the more evenly the pieces
    // fill the 608 pipes (us a step, best shape of two nodes per lane / this one: 128^2 7.2 / 4.5, 256^2
    // 11.2 / 10.0, 500x1000 59.5 / 56.6, 700^2 55.8 / 54.6, 2048^2 435.5 / 435.3).
    if (dtype == 0) return 5;
    // Other types: tiles in shared memory while the grid is small enough that a step is mostly launch and
    // latency (us a step, best other shape / tiles: f32s 250^2 1.9 / 1.4, 500^2 3.4 / 2.9, 900^2 7.4 / 7.0,
    // 1000^2 8.0 / 8.4; f32 128^2 1.8 / 1.3, 250^2 2.1 / 1.7, 300^2 2.2 / 2.6; q16s 500^2 5.9 / 5.0, 1050x1000
    // 16.7 / 16.0, 1200x1000 17.8 / 17.7; f16s 500x1000 7.1 / 5.3, 1200x1000 10.3 / 10.2, 1200^2 11.6 / 12.0).
    if (n < (dtype == 1 ? 90000 : (dtype == 2 ? 950000 : 1200000))) return kTileConfig;
    // f16s 2048^2 26.5 with shape 2, 27.5 with 0; 4096^2 100.3, 95.6
    if (dtype >= 3) return dtype == kDtypeQ16S || n < 8000000 ? 2 : 0;
    // f32, shapes 0 / 2: 500x1000 6.2 / 5.8, 900^2 8.3 / 8.1, 1000^2 9.4 / 9.6
    if (dtype == 1 && n < 950000) return 2;
    // Steps fused in the march: f32s from there on, f32 once the two population buffers outgrow the L2 cache
    // (below that the rows that neighbouring segments compute twice cost more than the saved launches).  Where a
    // strip's 120 columns are filled to less than 1 / 1.4 the tiles' 24 are the better cut.  us a step, march /
    // tiles / best row shape, columns filled: f32s 1200^2 (1.0) 10.3 / 13.5 / 12.9, 361x5000 (1 / 1.33) 14.6 / 17.8
    // / 21.6, 361x3000 10.5 / 9.9 / 10.0, 160x8000 (1 / 1.5) 14.8 / 12.7 / 13.1, 121x20000 (1 / 1.98) 27.2 / 24.9 /
    // 30.9; f32 1500x1200 16.4 / 20.1 / 18.4, 361x5000 21.2 / 21.4 / 21.5, 121x20000 41.6 / 31.0 / 31.5.
    const int filled = march_columns(nx);
    if (dtype == 2 || n >= 1600000) return 7ll * nx >= 5ll * filled ? kMarchConfig : kTileConfig;
    // f32 between: loads that leave L1 alone, shapes 0 / 5: 1000^2 9.4 / 9.4, 1150x1100 11.5 / 11.1, 1200^2 15.2 / 13.4,
    // 1300x1200 17.6 / 15.5 (march 14.9); a row that fills little of a warp's 64 nodes takes tiles (20x60000 55.6, 19.6)
    return nx < 40 ? kTileConfig : 5;
}

StepGeometry step_geometry(int dtype, int cfg, int nx, int ny) {
    StepGeometry g{};
    const Shape s = kShapes[dtype == 0 ? 0 : (storage_bytes(dtype) == 2 ? 2 : 1)][row_config(dtype, cfg)];
    g.grid_x = (nx + 32 * s.V - 1) / (32 * s.V);
    g.grid_y = (ny + s.BY * s.R - 1) / (s.BY * s.R);
    g.blocks = g.grid_x * g.grid_y;
    return g;
}

cudaError_t launch_step(int dtype, int cfg, const StepArgs& a, bool reduce, cudaStream_t st) {
    if (cfg < 0 || cfg >= kStepConfigs) return cudaErrorInvalidValue;
    cfg = row_config(dtype, cfg);
    switch (dtype) {
        case 0: return launch_step_f64(cfg, a, reduce, st);
        case 1: return launch_step_f32(cfg, a, reduce, st);
        case 2: return launch_step_f32s(cfg, a, reduce, st);
        case 3: return launch_step_f16s(cfg, a, reduce, st);
        case 4: return launch_step_bf16s(cfg, a, reduce, st);
        case 5: return launch_step_q16s(cfg, a, reduce, st);
        default: return cudaErrorInvalidValue;
    }
}

// Sum the per-block partials in a fixed order and publish the checkpoint (Eq. 6, mass).
__global__ void __launch_bounds__(256) k_finalize_checkpoint(const double* __restrict__ partials,
                                                             int nblocks, double nodes,
                                                             DevState* st) {
    __shared__ double sh[3][256];
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += 256) {
        s0 += partials[3ll * b];
        s1 += partials[3ll * b + 1];
        s2 += partials[3ll * b + 2];
    }
    sh[0][threadIdx.x] = s0;
    sh[1][threadIdx.x] = s1;
    sh[2][threadIdx.x] = s2;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
#pragma unroll
            for (int c = 0; c < 3; ++c) sh[c][threadIdx.x] += sh[c][threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        st->num = sh[1][0];
        st->den = sh[2][0];
        st->residual = sqrt(sh[1][0] / sh[2][0]);
        st->mass = nodes + sh[0][0];
        // LBM_Q16S: the checkpoint step stored against rho_ref[1]; the next one stores against
        // the mean density deviation just measured (unused by the other storage types)
        st->rho_ref[0] = st->rho_ref[1];
        if (isfinite(st->mass)) st->rho_ref[1] = st->mass / nodes - 1.0;
        st->base += kInterval;
        st->at_step = st->base;
        st->valid = 1;
    }
}

cudaError_t launch_finalize_checkpoint(const double* partials, int nblocks, double nodes,
                                       DevState* st, cudaStream_t s) {
    k_finalize_checkpoint<<<1, 256, 0, s>>>(partials, nblocks, nodes, st);
    return cudaGetLastError();
}

}  // namespace lbm
