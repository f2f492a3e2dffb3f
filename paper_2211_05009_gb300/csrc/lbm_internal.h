// lbm_internal.h -- declarations shared by the translation units of the CUDA library
// (kernel launchers and the per-context state).  Not part of the public ABI.
#pragma once

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>  // header-only; the ranges cost nothing unless a profiler is attached

#include "lbm_device.cuh"

namespace lbm {

// NVTX range over the host side of one library call (named in nsys / ncu timelines).
struct NvtxRange {
    explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange&) = delete;
    NvtxRange& operator=(const NvtxRange&) = delete;
};

// For as long as it lives, this thread's captures do not forbid it calls that allocate or wait: a graph
// captured and instantiated inside a library call would otherwise invalidate a capture that the caller
// has under way on another stream.
struct CaptureApart {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    CaptureApart() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~CaptureApart() { cudaThreadExchangeStreamCaptureMode(&mode); }
    CaptureApart(const CaptureApart&) = delete;
    CaptureApart& operator=(const CaptureApart&) = delete;
};

struct StepGeometry {
    int grid_x, grid_y, blocks;
};

// Launch shapes of the time step; all give identical populations.  0..5: one step per launch (row
// step, lbm_step_kernel.cuh).  6: kMarchSteps plain steps per launch (lbm_march.cuh) for FP32
// storage; steps left over run as one shorter launch, checkpoint steps one by one.  The other types take
// their default row shape there: FP64 is bound by its pipe and LBM_Q16S by its code conversions; a march
// of binary16 was tried and not kept (converting a value at a time between steps, 178 GLUPS at 4096^2 and
// 150 at 2048^2 where the row step ran 178 and 168).
// 7: several steps per launch in shared-memory tiles (lbm_tile.cuh), for small grids of every type
// but FP64, whose pipe pays for nodes computed twice.
constexpr int kStepConfigs = 8, kRowConfigs = 6, kMarchConfig = 6, kTileConfig = 7;
constexpr int kMarchSteps = 4;
struct TilePlan {
    int ow, oh, steps;     // nodes a tile owns, steps per launch
    int shift_x, shift_y;  // tiles begin at -shift
};
TilePlan tile_plan(int nx, int ny);
inline bool march_dtype(int dtype) { return dtype == 1 || dtype == 2; }
// Plain steps per launch of a shape.
inline int config_steps(int dtype, int cfg, int nx, int ny) {
    if (cfg == kMarchConfig && march_dtype(dtype)) return kMarchSteps;
    if (cfg == kTileConfig && dtype != 0) return tile_plan(nx, ny).steps;
    return 1;
}
// Row shape of the single steps of shapes 6 and 7 (f64, f32, f32s, f16s, bf16s, q16s): the fastest at
// 2048 x 2048, where FP32 storage is fused and every step of f64 and 16-bit storage takes it.
inline int default_row_config(int dtype) {
    constexpr int k[6] = {5, 0, 0, 2, 2, 2};
    return (dtype >= 0 && dtype < 6) ? k[dtype] : 0;
}
// Row shape of the single steps of a shape.
inline int row_config(int dtype, int cfg) { return cfg < kRowConfigs ? cfg : default_row_config(dtype); }
// Columns that the march's strips of an nx-wide grid own together (lbm_march.cu).
int march_columns(int nx);
// Shape of a new context; lbm_autotune measures all of them on the caller's size.
int default_step_config(int dtype, int nx, int ny);

constexpr int kDtypeQ16S = 5;
// LBM_Q16S scale S_j of direction j for lid speed U: the largest code is (2 - 2^-13) S_j, and
// 2 S_j = the power of two at or above K_j w_j max(|U|, 0.01) with K = 2 (rest), 5 (axes),
// 11/2 (diagonals), above the largest deviations met in lid-driven cavities from Re 74 to 8000
// (flat 131 x 13 to 2048^2): |h_j| < 4.5 w_j U (axes), 5.0 w_j U (diagonals), 1.0 w_j U (rest)
// once the mean density is taken out.
double q16_scale(int j, double U);
QCodec q16_codec(double U);

// Geometry of the step launch for a shape (also the number of reduction partials).
StepGeometry step_geometry(int dtype, int cfg, int nx, int ny);

// Bytes of the arithmetic type (FP64 for FP64 storage, FP32 otherwise): the Eq. 6 snapshot type.
inline int arith_bytes(int dtype) { return dtype == 0 ? 8 : 4; }

// Row pitch (elements) for a storage type: a multiple of 32 lanes x 16 bytes.
long long row_pitch(int dtype, int nx);
int storage_bytes(int dtype);

cudaError_t launch_step(int dtype, int cfg, const StepArgs& a, bool reduce, cudaStream_t st);
// `steps` (1 .. kMarchSteps) plain steps from a.src to a.dst in one launch (march_dtype types only);
// sms: multiprocessors of the device.
cudaError_t launch_march(int dtype, const StepArgs& a, int steps, int sms, cudaStream_t st);
// The same in shared-memory tiles (all types but FP64), steps <= p.steps.
cudaError_t launch_tile(int dtype, const StepArgs& a, const TilePlan& p, int steps, cudaStream_t st);
// `steps` plain steps in one launch as shape cfg takes them.
inline cudaError_t launch_fused(int dtype, int cfg, const StepArgs& a, int steps, int sms, cudaStream_t st) {
    return cfg == kTileConfig ? launch_tile(dtype, a, tile_plan(a.nx, a.ny), steps, st) : launch_march(dtype, a, steps, sms, st);
}
cudaError_t launch_finalize_checkpoint(const double* partials, int nblocks, double nodes,
                                       DevState* st, cudaStream_t s);

struct FieldArgs {
    void* f;  // populations [9][ny][pitch] of the storage type
    int nx, ny;
    long long pitch, plane;
    double U;
    int corner_moving;
    QCodec q;              // LBM_Q16S scales
    const DevState* st;    // LBM_Q16S reference density (rho_ref[0])
};

// f = f^eq(1, u0) with the Sec. 2.2 (i) initial velocity; snapshot = u0.
cudaError_t launch_init(int dtype, const FieldArgs& a, void* snap, cudaStream_t st);
// f = f^eq(rho, u) from dense [ny][nx] FP64 fields; snapshot = u.  neq_tau > 0 adds
// (1 - 1/tau) times the first-order Chapman-Enskog non-equilibrium part (tau = neq_tau).
cudaError_t launch_set_moments(int dtype, const FieldArgs& a, const double* rho, const double* ux,
                               const double* uy, void* snap, double neq_tau, cudaStream_t st);
// Dense [ny][nx] FP64 moments (any output may be null).
cudaError_t launch_moments(int dtype, const FieldArgs& a, double* rho, double* ux, double* uy,
                           cudaStream_t st);
// Dense [9][ny][nx] FP64 populations <-> storage.
cudaError_t launch_get_populations(int dtype, const FieldArgs& a, double* out, cudaStream_t st);
cudaError_t launch_set_populations(int dtype, const FieldArgs& a, const double* in, cudaStream_t st);
// Mass: sum over nodes of (rho - 1) into partials, then N + sum into st->scalar.
cudaError_t launch_mass(int dtype, const FieldArgs& a, double* partials, int max_partials,
                        DevState* state, cudaStream_t st);
// Stream function (u_x = dPsi/dy, trapezoid in y from Psi = 0 at y = 0) with window extrema
// into state->ext; psi (dense [ny][nx]) may be null.  scratch needs psi_scratch_doubles().
size_t psi_scratch_doubles(int nx, int ny);
cudaError_t launch_stream_function(int dtype, const FieldArgs& a, double* psi, int i0, int i1,
                                   int j0, int j1, double* scratch, DevState* state,
                                   cudaStream_t st);

}  // namespace lbm
