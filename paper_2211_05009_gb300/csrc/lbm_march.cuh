// lbm_march.cuh -- T time steps of the D2Q9 cavity in one pass over memory (FP32 arithmetic).
//
// 2048^2 LBM_F32S, T = 4: 21.8 us a step (192 GLUPS) against 46.6 (90) of the row step, which HBM
// bounds at 94; 4096^2 76 against 175 us; LBM_F32 2048^2 30.9 against 46.6.  What bounds it now is the FP32
// pipe: 61 packed operations a node, 15 % more of them for rows and 7 % for columns computed twice, take two thirds of the time,
// register moves that pairs need most of the rest (336 instructions per 128 nodes and step).
//
// A step of its own reads and writes every population once (18 values a node), which is what bounds
// the row step on grids beyond the L2 cache and leaves a launch per step on small ones.  Here a warp
// takes a strip of columns and a segment of rows and marches up the rows with all T steps in
// flight: step 1 reads row sets from memory, step l + 1 consumes the rows that step l has just
// produced, one row behind it, and only step T writes.  Between two steps a warp keeps what the pull
// of the next one still needs, in the storage format (so that T fused steps are bitwise T single
// ones): directions 2, 5, 6 (c_y = +1) of the last two rows and 0, 1, 3 of the last one, nine values
// a node, in its own part of shared memory, each lane its own nodes (no barrier).  In registers they
// would have to change places every row, which wants the row loop and the step loop unrolled:
// measured, the unrolled kernel outgrows the instruction cache (2048^2, T = 4, no packed arithmetic in
// either: 47 us a step unrolled, 30 us in this form).  Directions 4, 7, 8 of the newest row
// stay in registers.
//
// Lanes own V consecutive nodes; the x neighbours come by warp shuffle, so each step spoils one more
// node at both ends of the strip: H = ceil(T/V) lanes on each side only feed their neighbours, and
// strips overlap by them.  In y, step l of a segment [y0, y1) covers rows y0 - (T - l) .. y1 - 1 +
// (T - l).  Nodes k and k + V/2 of a lane form a pair, on which the packed FP32 instructions work;
// with that pairing the shift by one node renames pairs except at one end.
//
// Walls: a ring node is the collided inner neighbour plus a difference of equilibria (wall_shift),
// so row 0 comes with row 1 from the same pulled values; row ny - 1 takes one more pass over the
// values pulled for row ny - 2.
#pragma once

#include "lbm_step_kernel.cuh"

namespace lbm {

// V populations of one direction as V/2 pairs (nodes k, k + V/2): `Mem` is their layout in memory, `Ring`
// that between two fused steps, a pair as it lies in registers.  LBM_F32 is rounded to f = g + w wherever a
// step of its own would store it.
template <bool SHIFTED, int V>
struct RowCodec {
    static constexpr int HV = V / 2;
    using Mem = typename Raw<V * 4>::T;
    using Ring = typename Raw<8>::T;
    __device__ static __forceinline__ f32x2 in(f32x2 p, int j) { return SHIFTED ? p : rsub(p, f32x2(wd(j))); }
    __device__ static __forceinline__ f32x2 out(f32x2 p, int j) { return SHIFTED ? p : radd(p, f32x2(wd(j))); }
    __device__ static __forceinline__ void load(Mem r, int j, f32x2 (&p)[HV]) {
        union { Mem u; float s[V]; } b;
        b.u = r;
#pragma unroll
        for (int k = 0; k < HV; ++k) p[k] = in(f32x2(b.s[k], b.s[k + HV]), j);
    }
    __device__ static __forceinline__ Mem store(const f32x2 (&p)[HV], int j) {
        union { Mem u; float s[V]; } b;
#pragma unroll
        for (int k = 0; k < HV; ++k) {
            const f32x2 v = out(p[k], j);
            b.s[k] = v.lo();
            b.s[k + HV] = v.hi();
        }
        return b.u;
    }
    // one direction of a ring row: pair k of lane l at word 32 k + l
    __device__ static __forceinline__ void get(const Ring* r, int j, f32x2 (&p)[HV]) {
#pragma unroll
        for (int k = 0; k < HV; ++k) {
            union { Ring u; float s[2]; } b;
            b.u = r[32 * k];
            p[k] = in(f32x2(b.s[0], b.s[1]), j);
        }
    }
    __device__ static __forceinline__ void put(Ring* r, const f32x2 (&p)[HV], int j) {
#pragma unroll
        for (int k = 0; k < HV; ++k) {
            const f32x2 v = out(p[k], j);
            union { Ring u; float s[2]; } b;
            b.s[0] = v.lo();
            b.s[1] = v.hi();
            r[32 * k] = b.u;
        }
    }
    // what put and get make of values that stay in registers
    __device__ static __forceinline__ void round(int j, f32x2 (&p)[HV]) {
        if constexpr (!SHIFTED) {
#pragma unroll
            for (int k = 0; k < HV; ++k) p[k] = in(out(p[k], j), j);
        }
    }
};

template <int V, int T>
struct StripGeometry {
    static constexpr int kHalo = (T + V - 1) / V;         // lanes at each end that only feed neighbours
    static constexpr int kWidth = (32 - 2 * kHalo) * V;   // columns a strip owns
    // The right wall takes its inner neighbour's pulled values, so it may not be the only column of
    // the last strip (T = V leaves no halo column to spare): the strips then begin V columns earlier.
    __host__ __device__ static int shift(int nx) { return (nx - 1) % kWidth == 0 ? V : 0; }
    __host__ __device__ static int strips(int nx) { return (nx + shift(nx) + kWidth - 1) / kWidth; }
    // first column of a strip's lanes
    __host__ __device__ static int begin(int strip, int nx) { return strip * kWidth - kHalo * V - shift(nx); }
};

// Values of V nodes that a warp keeps between two steps: 0, 1, 3 of the newest row, 2, 5, 6 of the
// last two.
constexpr int kRingRows = 9;
template <typename S, int V, int T>
constexpr int march_ring_bytes() { return (T - 1) * kRingRows * 32 * V * (int)sizeof(S); }

__device__ __forceinline__ float pair_get(const f32x2& p, int h) { return h ? p.hi() : p.lo(); }

// Advance rows [y0, y1) of the strip whose lanes begin at column xs by `steps` <= T steps (FULL: by T) from src to dst.  y1 - y0
// >= 2.  t0 = global index of the state in src.  ring_v: march_ring_bytes of shared memory of this
// warp's own.
template <typename S, bool SHIFTED, int V, int T, bool FULL, int HINT, typename Probes>
__device__ __forceinline__ void march(const S* __restrict__ src, S* __restrict__ dst, const CavityView<float>& cv,
                                      int lane, int xs, int y0, int y1, int steps, const Probes& probes, long long t0,
                                      void* ring_v) {
    using Codec = RowCodec<SHIFTED, V>;
    static_assert(sizeof(S) == 4, "FP32 storage");
    using Mem = typename Codec::Mem;
    using Ring = typename Codec::Ring;
    using G = StripGeometry<V, T>;
    const int n = FULL ? T : steps;
    constexpr int HV = V / 2, kRow = 32 * HV;  // ring words of one direction
    const int nx = cv.nx, ny = cv.ny;
    const long long pitch = cv.pitch, plane = cv.plane;
    const Relax<float> rs = make_relax<float>(cv.omega);
    const Relax<f32x2> rx{f32x2(rs.ow1), f32x2(rs.ow5), f32x2(rs.w4), f32x2(rs.w9),
                          f32x2(rs.pw9), f32x2(rs.khalf), f32x2(rs.nhalf), f32x2(rs.o12)};
    const Omega<f32x2> om = make_omega<f32x2>(cv.omega);
    const f32x2 one_ref(1.0f);
    const int x0 = xs + lane * V;
    const bool own = lane >= G::kHalo && lane < 32 - G::kHalo && x0 >= 0 && x0 < nx;
    const bool edge = xs <= 0 || xs + 32 * V >= nx;  // the warp holds a wall column or padding
    const long long xl = min((long long)max(x0, 0), pitch - V);  // column loads stay in the row
    // observing points in this strip's own columns and in rows [y0, y1), of this lane and of any lane
    unsigned pmask = 0;
    for (int p = 0; p < probes.n(); ++p)
        if (own && probes.px(p) >= x0 && probes.px(p) < x0 + V && probes.py(p) >= y0 && probes.py(p) < y1) pmask |= 1u << p;
    const unsigned watch = __reduce_or_sync(kFull, pmask);
    // Only the rows around a point leave the plain path, decided once per row of step 1: the warp with the
    // most to do ends last, and the rest wait for it (2048^2, two points in one strip: 30.7 us a step with
    // every row of their segments on the other path, 22.6 so; 21.9 without points).  The batch and
    // LBM_F32 decide once per segment: their kernels have no register left for the rows (45 cavities 20.5
    // -> 20.8 ms; LBM_F32 2048^2 without points 31.3 -> 34.1 us a step).
    constexpr bool kByRow = SHIFTED && !std::is_same<Probes, ProbeOne>::value;
    bool sampled = !kByRow && watch;
    Ring* const ring = static_cast<Ring*>(ring_v) + lane;

    const int i0 = max(1, y0 - (n - 1)), i1 = y1 + n - 2;
    auto store_row = [&](int y, const f32x2 (&f)[9][HV]) {
        S* p = dst + (long long)y * pitch + x0;
#pragma unroll
        for (int j = 0; j < 9; ++j) {
            f32x2 v[HV];
#pragma unroll
            for (int k = 0; k < HV; ++k) v[k] = f[j][k];
            if (edge) {  // padding holds the rest state
#pragma unroll
                for (int k = 0; k < HV; ++k)
                    v[k] = f32x2(x0 + k < nx ? v[k].lo() : 0.0f, x0 + k + HV < nx ? v[k].hi() : 0.0f);
            }
            *reinterpret_cast<Mem*>(p + j * plane) = Codec::store(v, j);
        }
    };
    constexpr int kLines = (32 * V * (int)sizeof(S) + 127) / 128;  // 128-byte lines of a warp's row
    constexpr int kAhead = (9 * kLines + 31) / 32;
    const S* ahead[kAhead];
#pragma unroll
    for (int m = 0; m < kAhead; ++m) {
        const int q = min(lane + 32 * m, 9 * kLines - 1), j = q / kLines;
        const int dy = j == 2 || j == 5 || j == 6 ? 1 : (j == 4 || j == 7 || j == 8 ? -1 : 0);
        const long long x = min((long long)max(xs, 0) + q % kLines * (128 / (int)sizeof(S)), pitch - 1);
        ahead[m] = src + j * plane - dy * pitch + x;
    }
    // The nine rows that centre row i (ny - 2 for the top wall) pulls from.  The row above is
    // brought towards the L2 cache: the loads themselves are not prefetched (36 registers for V = 4),
    // the warp's siblings cover their latency.
    auto load_rows = [&](int i, f32x2 (&f)[9][HV]) {
        const S* p = src + (long long)min(i, ny - 2) * pitch + xl;
        Mem r[9];
#pragma unroll
        for (int j = 0; j < 9; ++j) r[j] = ldg_vec<Mem, HINT>(reinterpret_cast<const Mem*>(p + j * plane - cy(j) * pitch));
        if (i + 1 < min(i1 + 1, ny - 2)) {
            const long long up = (long long)(i + 1) * pitch;
#pragma unroll
            for (int m = 0; m < kAhead; ++m) asm volatile("prefetch.global.L2 [%0];" ::"l"(ahead[m] + up));
        }
#pragma unroll
        for (int j = 0; j < 9; ++j) Codec::load(r[j], j, f[j]);
    };

    // Pull (shift by c_x within the warp), moments, collision and walls of row y of step l; f: the
    // nine rows it pulls from in, the produced row out.
    auto advance_row = [&](int y, int l, int i, f32x2 (&f)[9][HV]) {
#pragma unroll
        for (int j = 0; j < 9; ++j) {
            if (cx(j) == 1) {
                const float left = __shfl_up_sync(kFull, f[j][HV - 1].hi(), 1);
                const f32x2 first(left, f[j][HV - 1].lo());
#pragma unroll
                for (int k = HV - 1; k > 0; --k) f[j][k] = f[j][k - 1];
                f[j][0] = first;
            } else if (cx(j) == -1) {
                const float right = __shfl_down_sync(kFull, f[j][0].lo(), 1);
                const f32x2 last(f[j][0].hi(), right);
#pragma unroll
                for (int k = 0; k < HV - 1; ++k) f[j][k] = f[j][k + 1];
                f[j][HV - 1] = last;
            }
        }
        if (xs <= 0) {  // the left wall takes the values pulled by its inner neighbour
#pragma unroll
            for (int j = 0; j < 9; ++j)
                f[j][0] = f32x2(x0 == 0 ? pair_get(f[j][1 % HV], HV == 1) : f[j][0].lo(), f[j][0].hi());
        }
        if (xs + 32 * V >= nx) {  // the right wall: slot sr of one lane, the same slot in every row
            const int sr = (nx - 1 - xs) % V;
            const bool mine = x0 + sr == nx - 1;
#pragma unroll
            for (int k = 0; k < V; ++k) {
                if (sr != k) continue;
#pragma unroll
                for (int j = 0; j < 9; ++j) {
                    float v;
                    if (k == 0) v = __shfl_up_sync(kFull, f[j][HV - 1].hi(), 1);
                    else v = pair_get(f[j][(k - 1) % HV], (k - 1) / HV);
                    f32x2& p = f[j][k % HV];
                    if (k < HV) p = f32x2(mine ? v : p.lo(), p.hi());
                    else p = f32x2(p.lo(), mine ? v : p.hi());
                }
            }
        }
        const bool top = y == ny - 1;
        const float wall_u = top ? cv.Ulid : 0.0f;  // of the nodes of row y that are walls but no corners
        float vx[V], vy[V];                         // velocities, for observing points
        // row 0, the wall below the values that row 1 pulls, for the next step's pull or the store
        auto emit_bottom = [&](const f32x2 (&w)[9][HV]) {
            if (l < n) {
                Ring* q = ring + ((l - 1) * kRingRows + 6 - 3 * (i & 1)) * kRow;
                Codec::put(q, w[2], 2);
                Codec::put(q + kRow, w[5], 5);
                Codec::put(q + 2 * kRow, w[6], 6);
            } else if (own && y0 == 0) {
                store_row(0, w);
            }
        };
        auto wall_speed = [&](int x) { return cv.corner_moving || (x > 0 && x < nx - 1) ? wall_u : 0.0f; };
        if constexpr (kOnPairs<S, SHIFTED>) {
            f32x2 rho[HV], ux[HV], uy[HV];
#pragma unroll
            for (int k = 0; k < HV; ++k) {
                f32x2 g[9], out[9], drho;
#pragma unroll
                for (int j = 0; j < 9; ++j) g[j] = f[j][k];
                collide<f32x2>(g, one_ref, rx, out, drho, rho[k], ux[k], uy[k]);
#pragma unroll
                for (int j = 0; j < 9; ++j) f[j][k] = out[j];
            }
            if (edge | top | sampled | (y == 1)) {  // a warp or a row with walls or observing points
#pragma unroll
                for (int k = 0; k < V; ++k) {
                    vx[k] = pair_get(ux[k % HV], k / HV);
                    vy[k] = pair_get(uy[k % HV], k / HV);
                }
                auto wall = [&](f32x2 (&w)[9][HV], int k, float W) {
                    const int h = k / HV, m = k % HV;
                    float out[9];
#pragma unroll
                    for (int j = 0; j < 9; ++j) out[j] = pair_get(w[j][m], h);
                    wall_shift<float>(pair_get(rho[m], h), vx[k], vy[k], W, out);
#pragma unroll
                    for (int j = 0; j < 9; ++j) w[j][m] = h ? f32x2(w[j][m].lo(), out[j]) : f32x2(out[j], w[j][m].hi());
                };
                if (y == 1) {
                    f32x2 w[9][HV];
#pragma unroll
                    for (int j = 0; j < 9; ++j)
#pragma unroll
                        for (int k = 0; k < HV; ++k) w[j][k] = f[j][k];
#pragma unroll
                    for (int k = 0; k < V; ++k) wall(w, k, 0.0f);
                    emit_bottom(w);
                }
#pragma unroll
                for (int k = 0; k < V; ++k) {
                    const int x = x0 + k;
                    if (!(top | (x == 0) | (x == nx - 1))) continue;
                    wall(f, k, wall_speed(x));
                    vx[k] = wall_speed(x);
                    vy[k] = 0.0f;
                }
            }
        } else {
            f32x2 rho[HV], drho[HV], ux[HV], uy[HV];
#pragma unroll
            for (int k = 0; k < HV; ++k) {
                f32x2 g[9];
#pragma unroll
                for (int j = 0; j < 9; ++j) g[j] = f[j][k];
                moments9(g, one_ref, drho[k], rho[k], ux[k], uy[k]);
            }
            const bool special = edge | top | sampled | (y == 1);
            if (special) {
#pragma unroll
                for (int k = 0; k < V; ++k) {
                    vx[k] = pair_get(ux[k % HV], k / HV);
                    vy[k] = pair_get(uy[k % HV], k / HV);
                }
            }
            // the wall node that takes the values slot k pulled
            auto wall = [&](int k, float W, float (&out)[9]) {
                const int h = k / HV, m = k % HV;
                float g[9];
#pragma unroll
                for (int j = 0; j < 9; ++j) g[j] = pair_get(f[j][m], h);
                wall9(g, pair_get(drho[m], h), pair_get(rho[m], h), vx[k], vy[k], W, cv.omega, out);
            };
            if (y == 1) {
                f32x2 w[9][HV];
#pragma unroll
                for (int m = 0; m < HV; ++m) {
                    float lo[9], hi[9];
                    wall(m, 0.0f, lo);
                    wall(m + HV, 0.0f, hi);
#pragma unroll
                    for (int j = 0; j < 9; ++j) w[j][m] = f32x2(lo[j], hi[j]);
                }
                emit_bottom(w);
            }
            if (edge | top) {  // wall nodes from the pulled values, the others as below
#pragma unroll
                for (int k = 0; k < HV; ++k) {
                    f32x2 g[9], out[9];
#pragma unroll
                    for (int j = 0; j < 9; ++j) g[j] = f[j][k];
                    collide9<kMomentum<S>>(g, drho[k], rho[k], ux[k], uy[k], om, out);
                    float wo[2][9];
                    bool is[2];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int x = x0 + k + h * HV;
                        is[h] = top | (x == 0) | (x == nx - 1);
                        if (!is[h]) continue;
                        wall(k + h * HV, wall_speed(x), wo[h]);
                        vx[k + h * HV] = wall_speed(x);
                        vy[k + h * HV] = 0.0f;
                    }
#pragma unroll
                    for (int j = 0; j < 9; ++j) f[j][k] = f32x2(is[0] ? wo[0][j] : out[j].lo(), is[1] ? wo[1][j] : out[j].hi());
                }
            } else {
#pragma unroll
                for (int k = 0; k < HV; ++k) {
                    f32x2 g[9], out[9];
#pragma unroll
                    for (int j = 0; j < 9; ++j) g[j] = f[j][k];
                    collide9<kMomentum<S>>(g, drho[k], rho[k], ux[k], uy[k], om, out);
#pragma unroll
                    for (int j = 0; j < 9; ++j) f[j][k] = out[j];
                }
            }
        }
        if (sampled) {
            for (int p = 0; p < probes.n(); ++p) {
                if (!((pmask >> p) & 1u)) continue;
                const bool low = y == 1 && probes.py(p) == 0;  // row 0 is at rest
                if (probes.py(p) != y && !low) continue;
                const long long t = t0 + l;
                const int ev = probes.every(p);
                long long m = t / ev - probes.start(p) / ev - 1;
                if (t % ev || m < 0) continue;
                m %= probes.cap(p);
                double px = 0.0, py = 0.0;
#pragma unroll
                for (int k = 0; k < V; ++k)
                    if (probes.px(p) == x0 + k && !low) {
                        px = double(vx[k]);
                        py = double(vy[k]);
                    }
                probes.series(p)[2 * m] = px;
                probes.series(p)[2 * m + 1] = py;
            }
        }
    };

    f32x2 row[9][HV];  // the row that the previous step has just produced
#pragma unroll 1
    for (int i = i0; i <= i1; ++i) {
        if constexpr (kByRow) {
            if (watch) {
                sampled = false;
                for (int p = 0; p < probes.n(); ++p)  // step l is at row i - l + 1; row 0 goes with row 1
                    if ((watch >> p) & 1u) sampled |= abs(2 * (i - max(probes.py(p), 1)) - n + 1) <= n + 1;
            }
        }
        bool on = i <= ny - 1;  // step 1 covers every row from i0 on
        if (on) {
            load_rows(i, row);
            advance_row(i, 1, i, row);
        }
#pragma unroll 1
        for (int l = 2; l <= n; ++l) {
            const int y = i - l + 1;
            Ring* z = ring + (l - 2) * kRingRows * kRow;  // directions 0, 1, 3 of row y of step l - 1
            Ring* p = z + (3 + 3 * (i & 1)) * kRow;       // 2, 5, 6 of row y - 1
            Ring* q = z + (6 - 3 * (i & 1)) * kRow;       // 2, 5, 6 of row y
            on = y >= max(1, y0 - n + l) && y <= ny - 1;
            f32x2 got[6][HV];
            Codec::get(z, 0, got[0]);
            Codec::get(z + kRow, 1, got[1]);
            Codec::get(z + 2 * kRow, 3, got[2]);
            Codec::get(p, 2, got[3]);
            Codec::get(p + kRow, 5, got[4]);
            Codec::get(p + 2 * kRow, 6, got[5]);
            if (y + 1 < ny - 1) {
                Codec::put(z, row[0], 0);
                Codec::put(z + kRow, row[1], 1);
                Codec::put(z + 2 * kRow, row[3], 3);
                Codec::put(p, row[2], 2);
                Codec::put(p + kRow, row[5], 5);
                Codec::put(p + 2 * kRow, row[6], 6);
            } else if (y + 1 == ny - 1) {
                // the top row has come in: keep what its inner row pulls for one more pass,
                // directions 4, 7, 8 in the slot that is no longer needed
#pragma unroll
                for (int m = 0; m < 3 * HV; ++m) q[32 * m] = p[32 * m];
                Codec::put(p, row[4], 4);
                Codec::put(p + kRow, row[7], 7);
                Codec::put(p + 2 * kRow, row[8], 8);
            } else {  // that pass: step l - 1 has ended (these are rounded already)
                Codec::get(q, 4, row[4]);
                Codec::get(q + kRow, 7, row[7]);
                Codec::get(q + 2 * kRow, 8, row[8]);
            }
            if (!on) continue;
#pragma unroll
            for (int k = 0; k < HV; ++k) {
                row[0][k] = got[0][k];
                row[1][k] = got[1][k];
                row[3][k] = got[2][k];
                row[2][k] = got[3][k];
                row[5][k] = got[4][k];
                row[6][k] = got[5][k];
            }
            Codec::round(4, row[4]);
            Codec::round(7, row[7]);
            Codec::round(8, row[8]);
            advance_row(y, l, i, row);
        }
        if (on && own && i - n + 1 >= y0) store_row(i - n + 1, row);
    }
}

// Warps of a launch: the first and the last strip, whose warps hold wall columns and take longer,
// have `esegs` segments each and come first, the strips between them `segs`.
struct MarchGrid {
    int strips, segs, esegs;
    __host__ __device__ int sides() const { return strips > 1 ? 2 : 1; }
    __host__ __device__ int warps() const { return sides() * esegs + (strips > 2 ? (strips - 2) * segs : 0); }
    // strip and rows of warp w in [0, warps())
    __device__ void place(int w, int ny, int& strip, int& y0, int& y1) const {
        int seg, of;
        const int s = sides();
        if (w < s * esegs) {
            of = esegs;
            seg = w / s;
            strip = w % s ? strips - 1 : 0;
        } else {
            of = segs;
            const int v = w - s * esegs;
            seg = v / (strips - 2);
            strip = 1 + v % (strips - 2);
        }
        y0 = (int)((long long)seg * ny / of);
        y1 = (int)((long long)(seg + 1) * ny / of);
    }
};

struct MarchArgs {
    StepArgs a;
    MarchGrid g;
    int n;  // steps
};

template <typename S, bool SHIFTED, int V, int T, bool FULL, int BY, int MINB>
__global__ void __launch_bounds__(32 * BY, MINB) k_march(const MarchArgs m) {
    extern __shared__ __align__(16) unsigned char march_smem[];
    const StepArgs& a = m.a;
    const int w = blockIdx.x * BY + threadIdx.y;
    if (w >= m.g.warps()) return;
    int strip, y0, y1;
    m.g.place(w, a.ny, strip, y0, y1);
    CavityView<float> cv;
    cv.nx = a.nx;
    cv.ny = a.ny;
    cv.pitch = a.pitch;
    cv.plane = a.plane;
    cv.omega = a.omega_f;
    cv.Ulid = a.U_f;
    cv.corner_moving = a.corner_moving;
    cv.sref = cv.sref_w = 0.0f;
    const long long t0 = a.probes.n ? a.state->base + a.s : 0;
    march<S, SHIFTED, V, T, FULL, 0>(static_cast<const S*>(a.src), static_cast<S*>(a.dst), cv, threadIdx.x,
                                     StripGeometry<V, T>::begin(strip, a.nx), y0, y1, m.n, ProbeList{a.probes}, t0, march_smem + threadIdx.y * march_ring_bytes<S, V, T>());
}

}  // namespace lbm
