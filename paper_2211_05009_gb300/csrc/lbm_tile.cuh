// lbm_tile.cuh -- several time steps of a small D2Q9 cavity per launch, in shared memory.
//
// On grids that fit the L2 cache a step of its own is a launch, a trip to L2 and one dependent chain
// (2 us at 128^2, 4 us at 500^2 for FP32 storage), whatever it computes: tiles take 1.0 and 2.8.  Here a block takes a tile of
// ow x oh nodes with a halo of n nodes on each side, copies it into shared memory in the storage
// format (so that n fused steps are bitwise n single ones) and takes n steps there, the computed
// region one node smaller on every side each time: the launch and the trip are paid once per n steps,
// for the halo's nodes computed by several blocks.  Two tile buffers in turn, one barrier per step.
// A tile with its halo is 32 columns wide: a lane is a column, and a warp takes two rows at a time,
// which the packed FP32 instructions work on together.
//
// A ring node pulls at its inner neighbour, up to two nodes away, which the halo covers as long as the
// wall column (row) is not the only one of a tile (tile_plan).
#pragma once

#include "lbm_step_kernel.cuh"

namespace lbm {

constexpr int kTileWarps = 8, kTileCols = 32;

struct TileArgs {
    StepArgs a;
    TilePlan p;
    int n;  // steps, <= p.steps
};

template <typename S, bool SHIFTED>
__global__ void __launch_bounds__(32 * kTileWarps, 2) k_tile(const TileArgs m) {
    using C = float;
    constexpr bool PAIRS = kOnPairs<S, SHIFTED>;
    extern __shared__ __align__(16) unsigned char tile_smem[];
    const StepArgs& a = m.a;
    const int n = m.n, nx = a.nx, ny = a.ny;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int hx = (kTileCols - m.p.ow) / 2, th = m.p.oh + 2 * n;  // hx >= n, a multiple of 4
    const int xs = (int)blockIdx.x * m.p.ow - m.p.shift_x - hx, ys = (int)blockIdx.y * m.p.oh - m.p.shift_y - n;
    const int area = kTileCols * th;
    S* buf = reinterpret_cast<S*>(tile_smem);
    S* nxt = buf + 9 * area;

    // copy the tile in: chunks of 4 nodes, all in flight; chunks outside the grid are never read
    for (int q = threadIdx.x; q < 8 * th; q += 32 * kTileWarps) {
        const int x = xs + (q & 7) * 4, y = ys + (q >> 3);
        if (y < 0 || y >= ny || x < 0 || x >= a.pitch) continue;
        const S* g = static_cast<const S*>(a.src) + (long long)y * a.pitch + x;
        const unsigned s = (unsigned)__cvta_generic_to_shared(buf + q * 4);
#pragma unroll
        for (int j = 0; j < 9; ++j)
            asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(s + (unsigned)(j * area * (int)sizeof(S))),
                         "l"(g + j * a.plane), "n"(4 * (int)sizeof(S)) : "memory");
    }
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
    const C omega = a.omega_f;
    const Relax<C> rs = make_relax<C>(omega);
    const Relax<f32x2> rx{f32x2(rs.ow1), f32x2(rs.ow5), f32x2(rs.w4), f32x2(rs.w9),
                          f32x2(rs.pw9), f32x2(rs.khalf), f32x2(rs.nhalf), f32x2(rs.o12)};
    const Omega<f32x2> om = make_omega<f32x2>(omega);
    C sref = C(0);
    if constexpr (kIsQ16<S>) sref = C(__ldcg(&a.state->rho_ref[0]));
    const C one_ref = kIsQ16<S> ? C(1.0) + sref : C(1.0);
    const long long t0 = a.probes.n ? a.state->base + a.s : 0;
    const int x = xs + lane;
    const bool wall_x = x == 0 || x == nx - 1;
    // gather column; lanes that never compute stay inside the buffer
    const int col = min(max(min(max(x, 1), nx - 2) - xs, 1), kTileCols - 2);
    __syncthreads();

    auto load = [&](const S* c, C (&g)[9]) {
#pragma unroll
        for (int j = 0; j < 9; ++j) {
            const S* p = c + j * area - cy(j) * kTileCols - cx(j);
            if constexpr (kIsQ16<S>) {
                g[j] = q16_decode(p->bits, a.q.dec[j]);
            } else {
                g[j] = St<S>::to(*p);
                if constexpr (!SHIFTED) g[j] -= C(wd(j));
            }
        }
    };
    auto store = [&](S* d, long long step, C (&out)[9]) {
#pragma unroll
        for (int j = 0; j < 9; ++j) {
            if constexpr (kIsQ16<S>) {
                bool sat = false;
                d[j * step].bits = (unsigned short)q16_encode(out[j], a.q.enc[j], sat);
            } else {
                if constexpr (!SHIFTED) out[j] += C(wd(j));
                d[j * step] = St<S>::from(out[j]);
            }
        }
    };
    // observing points among the nodes this lane's column owns
    unsigned points = 0;
    for (int k = 0; k < a.probes.n; ++k)
        if (a.probes.px[k] == x && lane >= hx && lane < kTileCols - hx && a.probes.py[k] >= ys + n &&
            a.probes.py[k] < ys + n + m.p.oh)
            points |= 1u << k;
    auto sample = [&](int y, int t, C ux, C uy) {
        for (int k = 0; k < a.probes.n; ++k) {
            if (!((points >> k) & 1u) || a.probes.py[k] != y) continue;
            const long long s = t0 + t;
            const int ev = a.probes.every[k];
            long long i = s / ev - a.probes.start[k] / ev - 1;
            if (s % ev || i < 0) continue;
            i %= a.probes.cap[k];
            a.probes.series[k][2 * i] = double(ux);
            a.probes.series[k][2 * i + 1] = double(uy);
        }
    };

#pragma unroll 1
    for (int t = 1; t <= n; ++t) {
        // rows and columns whose pulls are valid
        const int cy0 = max(ys + t, 0), cy1 = min(ys + th - t, ny);
        const bool act = lane >= hx - n + t && lane < kTileCols - hx + n - t && x >= 0 && x < nx;
        const bool last = t == n;
#pragma unroll 1
        for (int y = cy0 + 2 * warp; y < cy1; y += 2 * kTileWarps) {
            const int yb = min(y + 1, cy1 - 1);  // an odd last row is computed twice
            C g[2][9], out[2][9], drho[2], rho[2], ux[2], uy[2];
            load(buf + (min(max(y, 1), ny - 2) - ys) * kTileCols + col, g[0]);
            load(buf + (min(max(yb, 1), ny - 2) - ys) * kTileCols + col, g[1]);
            const bool wall[2] = {wall_x || y == 0 || y == ny - 1, wall_x || yb == 0 || yb == ny - 1};
            f32x2 gp[9], op[9], d, r, u, v;
#pragma unroll
            for (int j = 0; j < 9; ++j) gp[j] = f32x2(g[0][j], g[1][j]);
            if constexpr (PAIRS) {
                collide<f32x2>(gp, f32x2(1.0f), rx, op, d, r, u, v);
            } else {
                moments9(gp, f32x2(one_ref), d, r, u, v);
                collide9<kMomentum<S>>(gp, d, r, u, v, om, op);
            }
#pragma unroll
            for (int j = 0; j < 9; ++j) {
                out[0][j] = op[j].lo();
                out[1][j] = op[j].hi();
            }
            drho[0] = d.lo(), drho[1] = d.hi(), rho[0] = r.lo(), rho[1] = r.hi();
            ux[0] = u.lo(), ux[1] = u.hi(), uy[0] = v.lo(), uy[1] = v.hi();
            if (wall[0] | wall[1]) {
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    if (!wall[k]) continue;
                    const C W = ((k ? yb : y) == ny - 1) && (a.corner_moving || !wall_x) ? a.U_f : C(0);
                    if constexpr (PAIRS) wall_shift<C>(rho[k], ux[k], uy[k], W, out[k]);
                    else wall9(g[k], drho[k], rho[k], ux[k], uy[k], W, omega, out[k]);
                    ux[k] = W;
                    uy[k] = C(0);
                }
            }
            if (!act) continue;
            if (points) {
                sample(y, t, ux[0], uy[0]);
                if (yb != y) sample(yb, t, ux[1], uy[1]);
            }
            if (last) {
                S* d = static_cast<S*>(a.dst) + (long long)y * a.pitch + x;
                store(d, a.plane, out[0]);
                if (yb != y) store(d + a.pitch, a.plane, out[1]);
            } else {
                S* d = nxt + (y - ys) * kTileCols + lane;
                store(d, area, out[0]);
                if (yb != y) store(d + kTileCols, area, out[1]);
            }
        }
        __syncthreads();
        S* s = buf;
        buf = nxt;
        nxt = s;
    }
}

}  // namespace lbm
