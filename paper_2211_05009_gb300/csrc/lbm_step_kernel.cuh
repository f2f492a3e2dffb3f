// lbm_step_kernel.cuh -- the fused D2Q9 stream + collide + wall kernel (one launch per time step).
//
// Per node (Xiang & Shi, arXiv 2211.05009):
//   streaming   pull f_j(x - c_j) from the previous post-collision field        Eq. 1 (left)
//   moments     rho = sum f_j, rho u = sum c_j f_j                               Eq. 3
//   collision   f*_j = f_j + (f^eq_j - f_j)/tau                                   Eq. 1, Eq. 2
//   walls       ring nodes pull at their inner neighbour x_f instead and store
//               f^eq(rho_f, u_w) + (1 - 1/tau)(f(x_f) - f^eq(rho_f, u_f))           Sec. 2.2 (ii)
//               -- the non-equilibrium extrapolation rebuilt and collided in one go (the
//               rebuilt node has moments (rho_f, u_w), so its BGK step is this closed form).
// All arithmetic runs on deviations g_j = f_j - w_j, which keeps rounding relative to the flow
// rather than to the weights.  Every REDUCE launch (the 100th step of a checkpoint interval) also
// forms sum(rho - 1) and the two sums of Eq. 6 against the snapshot of 100 steps before, and writes
// the new snapshot: per node in the arithmetic type, per thread over its few nodes, and in FP64
// from the warp level up (FP64 throughput on this part is a small fraction of FP32's).
//
// Thread mapping: blockDim = (32, BY); each lane owns V consecutive nodes (FP64: 1; FP32: 2, an 8-byte
// vector, or 1 on small grids; 16-bit storage: 4, 8 bytes) of R consecutive rows, a warp 32*V nodes per
// row.  The row pitch is a multiple of 32*V for every launch shape, so all vector accesses are in
// bounds; the padding nodes (x >= nx) of the last strip that holds a node store the rest state, those
// beyond keep what they had, and no node reads either.
#pragma once

#include <type_traits>

#include "lbm_device.cuh"
#include "lbm_internal.h"

namespace lbm {

static constexpr unsigned kFull = 0xffffffffu;

template <int BYTES> struct Raw;
template <> struct Raw<16> { using T = uint4; };
template <> struct Raw<8> { using T = uint2; };
template <> struct Raw<4> { using T = unsigned int; };

// Vector load.  HINT 0: read-only path; 1: read-only with an L2 256-byte prefetch, no L1
// allocation; 2: coherent L2 load (ld.global.cg) for kernels that also write the array they read
// from across a grid barrier (the read-only path may serve stale lines there); 3: weak load cached
// in L1 (ld.global.ca) for the same kernels -- coherent because the loads follow the barrier's
// acquire, which discards the SM's stale L1 lines; spelled out in asm so that the compiler cannot
// turn it into a read-only-path load.
template <typename T, int HINT>
__device__ __forceinline__ T ldg_vec(const T* p) {
    if constexpr (HINT == 0) {
        return __ldg(p);
    } else if constexpr (HINT == 2) {
        return __ldcg(p);
    } else if constexpr (HINT == 3) {
        if constexpr (sizeof(T) == 16) {
            uint4 r;
            asm volatile("ld.global.ca.v4.u32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
            return r;
        } else if constexpr (sizeof(T) == 8) {
            uint2 r;
            asm volatile("ld.global.ca.v2.u32 {%0, %1}, [%2];" : "=r"(r.x), "=r"(r.y) : "l"(p));
            return r;
        } else {
            unsigned int r;
            asm volatile("ld.global.ca.u32 %0, [%1];" : "=r"(r) : "l"(p));
            return r;
        }
    } else if constexpr (sizeof(T) == 16) {
        uint4 r;
        asm volatile("ld.global.nc.L1::no_allocate.L2::256B.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
        return r;
    } else if constexpr (sizeof(T) == 8) {
        uint2 r;
        asm volatile("ld.global.nc.L1::no_allocate.L2::256B.v2.u32 {%0, %1}, [%2];"
                     : "=r"(r.x), "=r"(r.y) : "l"(p));
        return r;
    } else {
        unsigned int r;
        asm volatile("ld.global.nc.L1::no_allocate.L2::256B.u32 %0, [%1];" : "=r"(r) : "l"(p));
        return r;
    }
}

template <typename S, int V, int HINT = 0>
__device__ __forceinline__ void vload_n(const S* __restrict__ p, typename St<S>::C (&out)[V]) {
    using T = typename Raw<V * sizeof(S)>::T;
    union { T u; S s[V]; } b;
    b.u = ldg_vec<T, HINT>(reinterpret_cast<const T*>(p));
#pragma unroll
    for (int i = 0; i < V; ++i) out[i] = St<S>::to(b.s[i]);
}

// V values of a plain arithmetic-type array (the Eq. 6 snapshot), in 16-byte pieces.
template <typename C, int V, bool COHERENT = false>
__device__ __forceinline__ void cload(const C* p, C (&out)[V]) {
    constexpr int B = V * sizeof(C) < 16 ? V * sizeof(C) : 16;
    constexpr int PER = B / sizeof(C);
    using T = typename Raw<B>::T;
#pragma unroll
    for (int k = 0; k < V; k += PER) {
        union { T u; C c[PER]; } b;
        if constexpr (COHERENT)
            b.u = __ldcg(reinterpret_cast<const T*>(p + k));
        else
            b.u = *reinterpret_cast<const T*>(p + k);
#pragma unroll
        for (int i = 0; i < PER; ++i) out[k + i] = b.c[i];
    }
}
template <typename C, int V>
__device__ __forceinline__ void cstore(C* p, const C (&in)[V]) {
    constexpr int B = V * sizeof(C) < 16 ? V * sizeof(C) : 16;
    constexpr int PER = B / sizeof(C);
    using T = typename Raw<B>::T;
#pragma unroll
    for (int k = 0; k < V; k += PER) {
        union { T u; C c[PER]; } b;
#pragma unroll
        for (int i = 0; i < PER; ++i) b.c[i] = in[k + i];
        *reinterpret_cast<T*>(p + k) = b.u;
    }
}

template <typename S, int V>
__device__ __forceinline__ void vstore_n(S* __restrict__ p, const typename St<S>::C (&in)[V]) {
    using T = typename Raw<V * sizeof(S)>::T;
    union { T u; S s[V]; } b;
#pragma unroll
    for (int i = 0; i < V; ++i) b.s[i] = St<S>::from(in[i]);
    *reinterpret_cast<T*>(p) = b.u;
}

// Scalar load of one storage element, coherent at L2 when HINT == 2, L1-cached weak when 3.
template <typename S, int HINT>
__device__ __forceinline__ typename St<S>::C lds(const S* p) {
    if constexpr (HINT == 3) {
        if constexpr (sizeof(S) == 8) {
            unsigned long long r;
            asm volatile("ld.global.ca.u64 %0, [%1];" : "=l"(r) : "l"(p));
            union { unsigned long long u; S s; } b;
            b.u = r;
            return St<S>::to(b.s);
        } else if constexpr (sizeof(S) == 4) {
            unsigned int r;
            asm volatile("ld.global.ca.u32 %0, [%1];" : "=r"(r) : "l"(p));
            union { unsigned int u; S s; } b;
            b.u = r;
            return St<S>::to(b.s);
        } else {
            unsigned short r;
            asm volatile("ld.global.ca.u16 %0, [%1];" : "=h"(r) : "l"(p));
            union { unsigned short u; S s; } b;
            b.u = r;
            return St<S>::to(b.s);
        }
    } else if constexpr (HINT == 2) {
        if constexpr (sizeof(S) == 8) return St<S>::to(__ldcg(reinterpret_cast<const double*>(p)));
        else if constexpr (sizeof(S) == 4) return St<S>::to(__ldcg(reinterpret_cast<const float*>(p)));
        else {
            union { unsigned short u; S s; } b;
            b.u = __ldcg(reinterpret_cast<const unsigned short*>(p));
            return St<S>::to(b.s);
        }
    } else {
        return St<S>::to(*p);
    }
}

// One raw 16-bit element with the load path of HINT (see ldg_vec / lds).
template <int HINT>
__device__ __forceinline__ unsigned raw16(const void* p) {
    if constexpr (HINT == 3) {
        unsigned short r;
        asm volatile("ld.global.ca.u16 %0, [%1];" : "=h"(r) : "l"(p));
        return r;
    } else if constexpr (HINT == 2) {
        return __ldcg(static_cast<const unsigned short*>(p));
    } else {
        return *static_cast<const unsigned short*>(p);
    }
}

// One population value in the arithmetic type; qd = the LBM_Q16S decode scale of its direction.
template <typename S, int HINT>
__device__ __forceinline__ typename St<S>::C ld1(const S* p, float qd) {
    if constexpr (kIsQ16<S>) return q16_decode(raw16<HINT>(p), qd);
    else return lds<S, HINT>(p);
}

// V values of one direction: load (decoding LBM_Q16S codes with qd) / store (encoding with qe).
template <typename S, int V, int HINT>
__device__ __forceinline__ void vload_g(const S* __restrict__ p, float qd, typename St<S>::C (&out)[V]) {
    if constexpr (kIsQ16<S>) {
        using T = typename Raw<V * 2>::T;
        union { T u; unsigned short c[V]; } b;
        b.u = ldg_vec<T, HINT>(reinterpret_cast<const T*>(p));
#pragma unroll
        for (int i = 0; i < V; ++i) out[i] = q16_decode(b.c[i], qd);
    } else {
        vload_n<S, V, HINT>(p, out);
    }
}
template <typename S, int V>
__device__ __forceinline__ void vstore_g(S* __restrict__ p, float qe, const typename St<S>::C (&in)[V], bool& sat) {
    if constexpr (kIsQ16<S>) {
        using T = typename Raw<V * 2>::T;
        union { T u; unsigned short c[V]; } b;
#pragma unroll
        for (int i = 0; i < V; ++i) b.c[i] = (unsigned short)q16_encode(in[i], qe, sat);
        *reinterpret_cast<T*>(p) = b.u;
    } else {
        vstore_n<S, V>(p, in);
    }
}

// Pull one population row segment: out[i] = value at (x0 + i - DX), DX = c_x of the direction.
template <typename S, bool SHIFTED, int V, int DX, int HINT>
__device__ __forceinline__ void pull_row(const S* __restrict__ p, int lane, int x0, long long pitch,
                                         typename St<S>::C wj, float qd, typename St<S>::C (&out)[V]) {
    using C = typename St<S>::C;
    C v[V];
    vload_g<S, V, HINT>(p, qd, v);
    if constexpr (DX == 0) {
#pragma unroll
        for (int i = 0; i < V; ++i) out[i] = v[i];
    } else if constexpr (DX == 1) {
        C left = __shfl_up_sync(kFull, v[V - 1], 1);
        if (lane == 0) left = (x0 > 0) ? ld1<S, HINT>(p - 1, qd) : v[0];
        out[0] = left;
#pragma unroll
        for (int i = 1; i < V; ++i) out[i] = v[i - 1];
    } else {
        C right = __shfl_down_sync(kFull, v[0], 1);
        if (lane == 31) right = (x0 + V < pitch) ? ld1<S, HINT>(p + V, qd) : v[V - 1];
#pragma unroll
        for (int i = 0; i < V - 1; ++i) out[i] = v[i + 1];
        out[V - 1] = right;
    }
    if constexpr (!SHIFTED) {
#pragma unroll
        for (int i = 0; i < V; ++i) out[i] -= wj;
    }
}

// ------------------------------------------------------------------ arithmetic on pairs and momentum
// LBM_F64 and LBM_F32S.  The rounding of each operation is spelled out: every kernel that advances
// a node (row step, batch, fused march) must give bitwise the same populations, so none of them may
// leave the choice of contractions to the compiler.
__device__ __forceinline__ float radd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float rsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float rmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float rfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double radd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double rsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double rmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double rfma(double a, double b, double c) { return __fma_rn(a, b, c); }

// Two FP32 values in one 64-bit register pair, for Blackwell's packed FP32 instructions: the same
// roundings as the scalar ones at half the issue slots.
struct f32x2 {
    unsigned long long v;
    __device__ __forceinline__ f32x2() {}
    __device__ __forceinline__ f32x2(float lo, float hi) { asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi)); }
    __device__ __forceinline__ explicit f32x2(double c) : f32x2(float(c), float(c)) {}
    __device__ __forceinline__ explicit f32x2(float c) : f32x2(c, c) {}
    __device__ __forceinline__ float lo() const { return __uint_as_float((unsigned)v); }
    __device__ __forceinline__ float hi() const { return __uint_as_float((unsigned)(v >> 32)); }
};
__device__ __forceinline__ f32x2 radd(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f32x2 rsub(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f32x2 rmul(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f32x2 rfma(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}

// -1/v.
template <typename C>
__device__ __forceinline__ C nrcp(C v);
// FP32: hardware reciprocal estimate refined by one Newton-Raphson step r + r(1 - v r) (error
// below one ulp for the densities rho ~ 1 met here; no subnormals).  The IEEE-rounded reciprocal
// costs several times the instructions in a kernel that is partly issue-bound.
template <> __device__ __forceinline__ float nrcp<float>(float v) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(-v));
    return __fmaf_rn(r, __fmaf_rn(v, r, 1.0f), r);
}
template <> __device__ __forceinline__ f32x2 nrcp<f32x2>(f32x2 v) {
    float r0, r1;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(-v.lo()));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r1) : "f"(-v.hi()));
    const f32x2 r(r0, r1);
    return rfma(r, rfma(v, r, f32x2(1.0f)), r);
}
// FP64: hardware estimate of 1/v (20 leading bits in, 20 out: relative error within 2^-19) refined by one
// third-order step of Householder's family, r (1 + e + e^2) with e = 1 - v r: the error e^3 is within
// 2^-57, so three FP64 operations give 1/v to the nearest value or the one beside it.  Densities are near 1
// here; an infinity or NaN comes out as NaN, which the checkpoint reports.  `one` is 1 in a register.
__device__ __forceinline__ double nrcp(double v, double one) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(v));
    const double e = __fma_rn(-v, r, one);
    return __fma_rn(-r, __fma_rn(e, e, e), -r);
}

// The FP64 pipe takes 16.8 cycles for a warp's fused multiply-add of three registers and 19.9 for an
// addition, a product, or a multiply-add with a literal or kernel-parameter operand (measured, 4 to 28
// warps per SM).  So sums and products of the FP64 collision are multiply-adds by 1 and of -0, which
// round to the same values, and every constant sits in a register: 500 x 1000 56.2 -> 52.2 us a step,
// 2048^2 434 -> 402.
template <typename C>
struct Ops {
    const Relax<C>& k;
    __device__ __forceinline__ C add(C a, C b) const {
        if constexpr (std::is_same<C, double>::value) return rfma(a, k.one, b);
        else return radd(a, b);
    }
    __device__ __forceinline__ C sub(C a, C b) const {
        if constexpr (std::is_same<C, double>::value) return rfma(-b, k.one, a);
        else return rsub(a, b);
    }
    __device__ __forceinline__ C mul(C a, C b) const {
        if constexpr (std::is_same<C, double>::value) return rfma(a, b, k.nzero);
        else return rmul(a, b);
    }
};

// A parameter in a register: a value that went through a shuffle is no longer known to be uniform, so
// the compiler keeps it where a lane's own values are.
__device__ __forceinline__ Relax<double> in_registers(const Relax<double>& p) {
    Relax<double> k;
    auto own = [](double v) { return __shfl_sync(kFull, v, 0); };
    k.ow1 = own(p.ow1);
    k.ow5 = own(p.ow5);
    k.w4 = own(p.w4);
    k.w9 = own(p.w9);
    k.khalf = own(p.khalf);
    k.nhalf = own(p.nhalf);
    k.o12 = own(p.o12);
    k.m1 = own(p.m1);
    k.one = own(p.one);
    k.nzero = own(p.nzero);
    k.c15 = own(p.c15);
    k.cm3 = own(p.cm3);
    k.wall = p.wall;
    return k;
}

// Collision constants in FP32 (the FP64 ones come from the host, relax_f64).
template <typename C>
__device__ __forceinline__ Relax<C> make_relax(C omega) {
    Relax<C> k;
    k.ow1 = rmul(omega, C(1.0 / 9.0));
    k.ow5 = rmul(omega, C(1.0 / 36.0));
    k.w4 = rmul(k.ow1, C(-4.5));
    k.w9 = rmul(k.ow5, C(-9.0));
    k.pw9 = -k.w9;
    k.khalf = rmul(rsub(C(1.0), omega), C(0.5));
    k.nhalf = rmul(omega, C(-0.5));
    k.o12 = rmul(omega, C(1.0 / 12.0));
    return k;
}

// Moments (Eq. 3) and BGK collision (Eq. 1, Eq. 2) of a fluid node on deviations g = f - w.
// Both forms work on the opposite pairs (j, jbar) = (1,3) (2,4) (5,7) (8,6) with sum s and
// difference d, on the momentum j = rho u and on a = j_x u_x, b = j_y u_y, c = j_x u_y; the
// equilibrium of a pair is w (q +- 3 c_j.j) with q = drho + 9/2 (c_j.u)(c_j.j) - 3/2 (a + b):
// q_1 = drho + 3a - 3/2 b, q_2 = drho + 3b - 3/2 a, q_5/8 = drho + 3(a + b) +- 9c.
//
// FP32 (LBM_F32S): 61 FP32 operations.  A pair leaves as u +- v, its
// relaxed half sum u = (1 - omega) s/2 + omega w q and half difference v = d/2 + delta,
// delta = omega/2 (d^eq - d) with d^eq_5 = (j_x + j_y)/6, d^eq_8 = (j_x - j_y)/6.  delta_1 and
// delta_2 are taken from delta_5 and delta_8 so that the increments carry no momentum, and the rest
// population takes what keeps the mass: in FP32 the rounding of weights and moments otherwise
// shifts both in the same direction every step.  (Relaxing each direction by itself, 53 operations,
// is 1e-5 U off after 1000 steps of 133x77 at Re 400, this form 1.5e-7 U, increments formed per
// direction with their momentum taken out 3.6e-7 U.)
//
// FP64: 54 FP64 operations (72.7 instructions with the equilibrium formed per direction): the pipe
// issues 2 lanes per clock and SM, so the operation count is the run time (2048^2: 7.3 GLUPS then, 10.4
// now, 0.94 of what the pipe takes for 54.1 instructions a node at 16.8 cycles).
// out = keep g + (omega g^eq) with the pair's omega g^eq from two fused multiply-adds.
//
// FP64 ring nodes: f^eq(rho, u_w) + (1 - omega)(g - f^eq(rho, u)) at a resting wall has the fluid's
// density terms and its velocity terms times (omega - 1)/omega, so `vel` (1 for a fluid node) turns
// one into the other for five operations, where wall_shift takes 38 on a pipe that is the bound.
template <typename C, bool WALLS = false>
__device__ __forceinline__ void collide(const C (&g)[9], C one_ref, const Relax<C>& k, C (&out)[9], C& drho,
                                        C& rho, C& ux, C& uy, C vel = C(1.0)) {
    constexpr bool F64 = std::is_same<C, double>::value;
    const Ops<C> o{k};
    // d1 = g1 - g3, d2 = g2 - g4, and the negated n5 = g7 - g5, n8 = g6 - g8
    const C s1 = o.add(g[1], g[3]), d1 = o.sub(g[1], g[3]);
    const C s2 = o.add(g[2], g[4]), d2 = o.sub(g[2], g[4]);
    const C s5 = o.add(g[5], g[7]), n5 = o.sub(g[7], g[5]);
    const C s8 = o.add(g[8], g[6]), n8 = o.sub(g[6], g[8]);
    drho = o.add(o.add(o.add(s1, s2), o.add(s5, s8)), g[0]);
    // -j and -1/rho, whose signs cancel in u: negations would be instructions of their own
    C jx = o.sub(o.add(n5, n8), d1);
    C jy = o.sub(o.sub(n5, n8), d2);
    C inv;
    if constexpr (F64) {
        rho = o.add(drho, k.one);
        inv = nrcp(rho, k.one);
    } else {
        rho = radd(one_ref, drho);
        inv = nrcp<C>(rho);
    }
    ux = o.mul(jx, inv);
    uy = o.mul(jy, inv);
    if constexpr (WALLS) {
        jx = o.mul(jx, vel);
        jy = o.mul(jy, vel);
    }
    // -a, -b, -c and -(a + b).  No sum of two products: the assembler fuses such packed ones.
    const C a = o.mul(jx, ux), b = o.mul(jy, uy), c = o.mul(jx, uy);
    const C ab = rfma(jx, ux, b);
    const C jp = o.add(jx, jy), jm = o.sub(jx, jy);
    C c15, cm3;
    if constexpr (F64) c15 = k.c15, cm3 = k.cm3;
    else c15 = C(1.5), cm3 = C(-3.0);
    const C base = rfma(c15, ab, drho);
    const C p1 = o.mul(k.ow1, base), p5 = o.mul(k.ow5, rfma(cm3, ab, drho));
    const C q1 = rfma(k.w4, a, p1), q2 = rfma(k.w4, b, p1);
    const C q5 = rfma(k.w9, c, p5);
    C q8;
    if constexpr (F64) q8 = rfma(-k.w9, c, p5);
    else q8 = rfma(k.pw9, c, p5);
    if constexpr (!F64) {
        const C u1 = rfma(k.khalf, s1, q1), u2 = rfma(k.khalf, s2, q2);
        const C u5 = rfma(k.khalf, s5, q5), u8 = rfma(k.khalf, s8, q8);
        const C e5 = rfma(k.nhalf, n5, rmul(k.o12, jp));  // -delta_5
        const C e8 = rfma(k.nhalf, n8, rmul(k.o12, jm));  // -delta_8
        const C v1 = rfma(C(0.5), d1, radd(e5, e8)), v2 = rfma(C(0.5), d2, rsub(e5, e8));
        const C v5 = rfma(C(0.5), n5, e5), v8 = rfma(C(0.5), n8, e8);  // negated
        out[0] = rfma(C(-2.0), radd(radd(u1, u2), radd(u5, u8)), drho);
        out[1] = radd(u1, v1);
        out[3] = rsub(u1, v1);
        out[2] = radd(u2, v2);
        out[4] = rsub(u2, v2);
        out[5] = rsub(u5, v5);
        out[7] = radd(u5, v5);
        out[8] = rsub(u8, v8);
        out[6] = radd(u8, v8);
    } else {
        const C m1 = k.m1, m5 = k.o12;
        out[0] = rfma(k.khalf, g[0], o.mul(k.nhalf, base));
        out[1] = rfma(k.khalf, g[1], rfma(-m1, jx, q1));
        out[3] = rfma(k.khalf, g[3], rfma(m1, jx, q1));
        out[2] = rfma(k.khalf, g[2], rfma(-m1, jy, q2));
        out[4] = rfma(k.khalf, g[4], rfma(m1, jy, q2));
        out[5] = rfma(k.khalf, g[5], rfma(-m5, jp, q5));
        out[7] = rfma(k.khalf, g[7], rfma(m5, jp, q5));
        out[8] = rfma(k.khalf, g[8], rfma(-m5, jm, q8));
        out[6] = rfma(k.khalf, g[6], rfma(m5, jm, q8));
    }
}

// Wall closure of a ring node whose inner neighbour x_f collided to `out` with moments (rho, u):
// f^eq(rho, u_w) + (1 - omega)(f(x_f) - f^eq(rho, u)) = out + f^eq(rho, u_w) - f^eq(rho, u), the
// difference of two equilibria of equal density: w (q +- 3 c_j.j) of the differences of a, b, c
// and j.  The walls rest or move along x with speed W.
template <typename C>
__device__ __forceinline__ void wall_shift(C rho, C ux, C uy, C W, C (&out)[9]) {
    const C jx = rmul(rho, ux), jy = rmul(rho, uy), jw = rmul(rho, W);
    const C a = rsub(rmul(jw, W), rmul(jx, ux)), b = rmul(-jy, uy), c = rmul(-jx, uy);
    const C mx = rmul(C(3.0), rsub(jw, jx)), my = rmul(C(-3.0), jy);
    const C ab = radd(a, b), c9 = rmul(C(9.0), c);
    const C q1 = rfma(C(-1.5), b, rmul(C(3.0), a)), q2 = rfma(C(-1.5), a, rmul(C(3.0), b));
    const C qd = rmul(C(3.0), ab), q5 = radd(qd, c9), q8 = rsub(qd, c9);
    const C mp = radd(mx, my), mm = rsub(mx, my);
    const C w1 = C(1.0 / 9.0), w5 = C(1.0 / 36.0);
    out[0] = rfma(C(-2.0 / 3.0), ab, out[0]);  // -3/2 w_0
    out[1] = rfma(w1, radd(q1, mx), out[1]);
    out[3] = rfma(w1, rsub(q1, mx), out[3]);
    out[2] = rfma(w1, radd(q2, my), out[2]);
    out[4] = rfma(w1, rsub(q2, my), out[4]);
    out[5] = rfma(w5, radd(q5, mp), out[5]);
    out[7] = rfma(w5, rsub(q5, mp), out[7]);
    out[8] = rfma(w5, radd(q8, mm), out[8]);
    out[6] = rfma(w5, rsub(q8, mm), out[6]);
}

// What a wall moving along x with speed W adds to a resting one: f^eq(rho, W) - f^eq(rho, 0).
template <typename C>
__device__ __forceinline__ void lid_shift(C rho, C W, C (&out)[9]) {
    const C j = rmul(rho, W), a = rmul(j, W);
    const C w1 = C(1.0 / 9.0), w5 = C(1.0 / 36.0);
    const C a3 = rmul(C(3.0), a), j3 = rmul(C(3.0), j);
    out[0] = rfma(C(-2.0 / 3.0), a, out[0]);  // -3/2 w_0
    out[1] = rfma(w1, radd(a3, j3), out[1]);
    out[3] = rfma(w1, rsub(a3, j3), out[3]);
    out[2] = rfma(C(-1.5) * w1, a, out[2]);
    out[4] = rfma(C(-1.5) * w1, a, out[4]);
    out[5] = rfma(w5, radd(a3, j3), out[5]);
    out[8] = rfma(w5, radd(a3, j3), out[8]);
    out[6] = rfma(w5, rsub(a3, j3), out[6]);
    out[7] = rfma(w5, rsub(a3, j3), out[7]);
}

// ------------------------------------------------------------------ arithmetic per direction
// LBM_F32 and 16-bit storage: what these store is rounded far above FP32 arithmetic on deviations
// (4e-6 of the velocity after 250 steps of a 500 x 1000 cavity in LBM_F32, 5e-4 in binary16), so
// their results are that rounding's noise.  They keep the arithmetic that forms every direction by
// itself, and with it their results bit for bit; the rounding of each operation is spelled out here
// too, in two spellings that round alike (rounding to nearest is symmetric).  Packed nodes (march,
// tiles): a negation is an instruction, so signs are placed where nothing is negated by itself.
// Single nodes (row step): operands take a sign for nothing, and the plain signs cost one product less
// and let the compiler order the chain better (us a step, packed spelling / this one: LBM_F32 300^2 4.3 /
// 3.8, 1000^2 9.9 / 9.4, binary16 1200^2 11.9 / 11.6, 1500^2 15.9 / 15.4).
template <typename C>
struct Omega {
    C om, nom;        // omega, -omega
    C ow0, ow1, ow5;  // omega w_j
};
template <typename C>
__device__ __forceinline__ Omega<C> make_omega(float w) {
    return Omega<C>{C(w), C(-w), C(rmul(w, float(4.0 / 9.0))), C(rmul(w, float(1.0 / 9.0))), C(rmul(w, float(1.0 / 36.0)))};
}

// Moments of a node (Eq. 3).
__device__ __forceinline__ void moments9(const f32x2 (&g)[9], f32x2 one_ref, f32x2& drho, f32x2& rho, f32x2& ux, f32x2& uy) {
    drho = radd(radd(radd(radd(g[0], g[1]), radd(g[2], g[3])), radd(radd(g[4], g[5]), radd(g[6], g[7]))), g[8]);
    rho = radd(one_ref, drho);
    const f32x2 inv = nrcp<f32x2>(rho);  // -1/rho, against -j
    ux = rmul(radd(radd(rsub(g[3], g[1]), rsub(g[6], g[5])), rsub(g[7], g[8])), inv);
    uy = rmul(radd(rsub(rsub(g[4], g[2]), radd(g[5], g[6])), radd(g[7], g[8])), inv);
}
__device__ __forceinline__ void moments9(const float (&g)[9], float one_ref, float& drho, float& rho, float& ux, float& uy) {
    drho = radd(radd(radd(radd(g[0], g[1]), radd(g[2], g[3])), radd(radd(g[4], g[5]), radd(g[6], g[7]))), g[8]);
    rho = radd(one_ref, drho);
    const float jx = radd(radd(rsub(g[1], g[3]), rsub(g[5], g[6])), rsub(g[8], g[7]));
    const float jy = rsub(radd(rsub(g[2], g[4]), radd(g[5], g[6])), radd(g[7], g[8]));
    const float inv = -nrcp<float>(rho);
    ux = rmul(jx, inv);
    uy = rmul(jy, inv);
}

// t_j with g^eq_j = w_j t_j, t_j = drho + rho A_j, A_j = 3 c.u + 9/2 (c.u)^2 - 3/2 u.u (Eq. 2).
__device__ __forceinline__ void eq_terms(f32x2 drho, f32x2 rho, f32x2 ux, f32x2 uy, f32x2 (&t)[9]) {
    const f32x2 nusq = rmul(f32x2(-1.5), rfma(ux, ux, rmul(uy, uy)));
    t[0] = rfma(rho, nusq, drho);
    auto pair = [&](int a, int b, f32x2 cu) {
        t[a] = rfma(rho, rfma(cu, rfma(f32x2(4.5), cu, f32x2(3.0)), nusq), drho);
        t[b] = rfma(rho, rfma(cu, rfma(f32x2(4.5), cu, f32x2(-3.0)), nusq), drho);
    };
    pair(1, 3, ux);
    pair(2, 4, uy);
    pair(5, 7, radd(ux, uy));
    pair(8, 6, rsub(ux, uy));
}
__device__ __forceinline__ void eq_terms(float drho, float rho, float ux, float uy, float (&t)[9]) {
    const float usq = rmul(1.5f, rfma(ux, ux, rmul(uy, uy)));
    t[0] = rfma(-rho, usq, drho);
    auto pair = [&](int a, int b, float cu) {
        t[a] = rfma(rho, rfma(cu, rfma(4.5f, cu, 3.0f), -usq), drho);
        t[b] = rfma(rho, rfma(-cu, rfma(4.5f, -cu, 3.0f), -usq), drho);
    };
    pair(1, 3, ux);
    pair(2, 4, uy);
    pair(5, 7, radd(ux, uy));
    pair(8, 6, rsub(ux, uy));
}

// Wall closure of a ring node from the values g pulled by its inner neighbour.
__device__ __forceinline__ void wall9(const float (&g)[9], float drho, float rho, float ux, float uy, float W, float omega,
                                      float (&out)[9]) {
    const float keep = rsub(1.0f, omega);  // 1 - 1/tau
    float t[9];
    eq_terms(drho, rho, ux, uy, t);
    // the wall's own terms, u = (W, 0): one each for c_x = 0, 1, -1
    const float usq = rmul(1.5f, rmul(W, W));
    const float w0 = rfma(-rho, usq, drho);
    const float wp = rfma(rho, rfma(W, rfma(4.5f, W, 3.0f), -usq), drho), wm = rfma(rho, rfma(-W, rfma(4.5f, -W, 3.0f), -usq), drho);
#pragma unroll
    for (int j = 0; j < 9; ++j)
        out[j] = rfma(float(wd(j)), cx(j) == 0 ? w0 : (cx(j) > 0 ? wp : wm), rmul(keep, rfma(-float(wd(j)), t[j], g[j])));
}

// The same closure with its contractions left to the compiler, which makes the ones spelled out above (the
// launch shapes' bitwise tests hold the tiles' walls against these).  For the row step in binary16 and
// bfloat16 alone: at its 64 registers the wall path decides which values spill, and of five spellings of it
// only this one leaves the interior path alone (binary16, us a step, this / the others: 1200^2 11.6 / 11.85
// .. 12.1, 2048^2 26.4 / 26.5 .. 28.1).
__device__ __forceinline__ void wall9_contracted(const float (&g)[9], float drho, float rho, float ux, float uy, float W,
                                                 float omega, float (&out)[9]) {
    auto equilibrium = [&](float vx, float vy, float (&e)[9]) {
        const float usq = 1.5f * (vx * vx + vy * vy);
        const float up = vx + vy, um = vx - vy;
        auto term = [&](float cu) { return drho + rho * (cu * (3.0f + 4.5f * cu) - usq); };
        e[0] = float(wd(0)) * (drho - rho * usq);
        e[1] = float(wd(1)) * term(vx);
        e[2] = float(wd(2)) * term(vy);
        e[3] = float(wd(3)) * term(-vx);
        e[4] = float(wd(4)) * term(-vy);
        e[5] = float(wd(5)) * term(up);
        e[6] = float(wd(6)) * term(-um);
        e[7] = float(wd(7)) * term(-up);
        e[8] = float(wd(8)) * term(um);
    };
    const float keep = 1.0f - omega;
    float e[9], ew[9];
    equilibrium(ux, uy, e);
    equilibrium(W, 0.0f, ew);
#pragma unroll
    for (int j = 0; j < 9; ++j) out[j] = ew[j] + keep * (g[j] - e[j]);
}

// Collision of a fluid node.  MOMENTUM: BGK as an increment d_j = (f^eq_j - f_j)/tau added to the
// pulled value, with the x and y momentum of d removed from the (1,3) and (2,4) pairs: in FP32 the
// rounding of f^eq otherwise shifts the momentum by a few ulps in the same direction every step.
// LBM_Q16S rounds its stores to nearest, which passes such a bias on unchanged on average, so it
// needs the correction as much as LBM_F32 does.  binary16 / bfloat16 swamp the bias and take the
// form per opposite pair, f*_j = g_j + omega (g^eq_j - g_j) with A = c2 +- 3 c.u.
template <bool MOMENTUM>
__device__ __forceinline__ void collide9(const f32x2 (&g)[9], f32x2 drho, f32x2 rho, f32x2 ux, f32x2 uy, const Omega<f32x2>& k,
                                         f32x2 (&out)[9]) {
    using C = f32x2;
    if constexpr (MOMENTUM) {
        C t[9], n[9];
        eq_terms(drho, rho, ux, uy, t);
#pragma unroll
        for (int j = 0; j < 9; ++j) n[j] = rfma(C(-wd(j)), t[j], g[j]);  // -d_j / omega
        const C d3 = rmul(k.nom, n[3]), d4 = rmul(k.nom, n[4]), d6 = rmul(k.nom, n[6]), d7 = rmul(k.nom, n[7]);
        // minus the x momentum, and the y momentum, of the increments
        const C nmx = radd(radd(rfma(k.om, n[1], d3), rfma(k.om, n[5], d6)), rfma(k.om, n[8], d7));
        const C my = rsub(rsub(rfma(k.nom, n[5], d6), rfma(k.om, n[2], d4)), rfma(k.nom, n[8], d7));
        out[0] = rfma(k.nom, n[0], g[0]);
        out[1] = radd(g[1], rfma(k.nom, n[1], rmul(C(0.5), nmx)));
        out[3] = radd(g[3], rfma(C(-0.5), nmx, d3));
        out[2] = radd(g[2], rfma(k.nom, n[2], rmul(C(-0.5), my)));
        out[4] = radd(g[4], rfma(C(0.5), my, d4));
        out[5] = rfma(k.nom, n[5], g[5]);
        out[8] = rfma(k.nom, n[8], g[8]);
        out[6] = radd(g[6], d6);
        out[7] = radd(g[7], d7);
    } else {
        const C nusq = rmul(C(-1.5), rfma(ux, ux, rmul(uy, uy)));
        const C r3 = rmul(C(3.0), rho), n3 = rmul(C(-3.0), rho);
        out[0] = rfma(k.ow0, rfma(rho, nusq, drho), rfma(k.nom, g[0], g[0]));
        auto pair = [&](int a, int b, C cu, C ow) {
            const C base = rfma(rho, rfma(rmul(C(4.5), cu), cu, nusq), drho);
            out[a] = rfma(ow, rfma(r3, cu, base), rfma(k.nom, g[a], g[a]));
            out[b] = rfma(ow, rfma(n3, cu, base), rfma(k.nom, g[b], g[b]));
        };
        pair(1, 3, ux, k.ow1);
        pair(2, 4, uy, k.ow1);
        pair(5, 7, radd(ux, uy), k.ow5);
        pair(8, 6, rsub(ux, uy), k.ow5);
    }
}
template <bool MOMENTUM>
__device__ __forceinline__ void collide9(const float (&g)[9], float drho, float rho, float ux, float uy, const Omega<float>& k,
                                         float (&out)[9]) {
    if constexpr (MOMENTUM) {
        float t[9], n[9];
        eq_terms(drho, rho, ux, uy, t);
#pragma unroll
        for (int j = 0; j < 9; ++j) n[j] = rfma(float(wd(j)), t[j], -g[j]);  // d_j / omega
        const float d3 = rmul(k.om, n[3]), d4 = rmul(k.om, n[4]), d6 = rmul(k.om, n[6]), d7 = rmul(k.om, n[7]);
        const float mx = radd(radd(rfma(k.om, n[1], -d3), rfma(k.om, n[5], -d6)), rfma(k.om, n[8], -d7));
        const float my = rsub(radd(rfma(k.om, n[2], -d4), rfma(k.om, n[5], d6)), rfma(k.om, n[8], d7));
        out[0] = rfma(k.om, n[0], g[0]);
        out[1] = radd(g[1], rfma(k.om, n[1], rmul(-0.5f, mx)));
        out[3] = radd(g[3], rfma(0.5f, mx, d3));
        out[2] = radd(g[2], rfma(k.om, n[2], rmul(-0.5f, my)));
        out[4] = radd(g[4], rfma(0.5f, my, d4));
        out[5] = rfma(k.om, n[5], g[5]);
        out[8] = rfma(k.om, n[8], g[8]);
        out[6] = radd(g[6], d6);
        out[7] = radd(g[7], d7);
    } else {
        const float usq = rmul(1.5f, rfma(ux, ux, rmul(uy, uy)));
        const float r3 = rmul(3.0f, rho);
        out[0] = rfma(k.ow0, rfma(-rho, usq, drho), rfma(-k.om, g[0], g[0]));
        auto pair = [&](int a, int b, float cu, float ow) {
            const float base = rfma(rho, rfma(rmul(4.5f, cu), cu, -usq), drho);
            out[a] = rfma(ow, rfma(r3, cu, base), rfma(-k.om, g[a], g[a]));
            out[b] = rfma(ow, rfma(-r3, cu, base), rfma(-k.om, g[b], g[b]));
        };
        pair(1, 3, ux, k.ow1);
        pair(2, 4, uy, k.ow1);
        pair(5, 7, radd(ux, uy), k.ow5);
        pair(8, 6, rsub(ux, uy), k.ow5);
    }
}

// Whether a storage type takes the arithmetic on pairs and momentum (collide, wall_shift).
template <typename S, bool SHIFTED> inline constexpr bool kOnPairs = SHIFTED && sizeof(S) >= 4;
// ... and whether its per-direction collision takes the momentum correction.
template <typename S> inline constexpr bool kMomentum = sizeof(S) == 4 || kIsQ16<S>;

// Streamed populations of one row segment (V nodes) of row y, walls folded in: wall rows gather
// at their inner row, the left/right wall nodes take the populations of x_f = 1 / nx - 2.
template <typename S, bool SHIFTED, int V, int HINT>
__device__ __forceinline__ void pull_segment(const S* __restrict__ src, int lane, int x0, int y, int nx,
                                             int ny, long long pitch, long long plane, const QCodec& q,
                                             typename St<S>::C (&f)[9][V]) {
    using C = typename St<S>::C;
    const int yc = min(max(y, 1), ny - 2);  // gather centre row
    if constexpr (V == 1) {
        // one node per lane: every lane gathers at its own x_f.  The three columns of a row share their
        // cache lines, and no load waits for a shuffle or sits in a branch.
        const S* pf = src + (long long)yc * pitch + min(max(x0, 1), nx - 2);
#pragma unroll
        for (int j = 0; j < 9; ++j) {
            vload_g<S, 1, HINT>(pf + j * plane - cy(j) * pitch - cx(j), q.dec[j], f[j]);
            if constexpr (!SHIFTED) f[j][0] -= C(wd(j));
        }
        return;
    }
    const S* pc = src + (long long)yc * pitch + x0;
    const S* ps = pc - pitch;  // row yc - 1: source of c_y = +1
    const S* pn = pc + pitch;  // row yc + 1: source of c_y = -1
    pull_row<S, SHIFTED, V, 0, HINT>(pc + 0 * plane, lane, x0, pitch, C(4.0 / 9.0), q.dec[0], f[0]);
    pull_row<S, SHIFTED, V, 1, HINT>(pc + 1 * plane, lane, x0, pitch, C(1.0 / 9.0), q.dec[1], f[1]);
    pull_row<S, SHIFTED, V, 0, HINT>(ps + 2 * plane, lane, x0, pitch, C(1.0 / 9.0), q.dec[2], f[2]);
    pull_row<S, SHIFTED, V, -1, HINT>(pc + 3 * plane, lane, x0, pitch, C(1.0 / 9.0), q.dec[3], f[3]);
    pull_row<S, SHIFTED, V, 0, HINT>(pn + 4 * plane, lane, x0, pitch, C(1.0 / 9.0), q.dec[4], f[4]);
    pull_row<S, SHIFTED, V, 1, HINT>(ps + 5 * plane, lane, x0, pitch, C(1.0 / 36.0), q.dec[5], f[5]);
    pull_row<S, SHIFTED, V, -1, HINT>(ps + 6 * plane, lane, x0, pitch, C(1.0 / 36.0), q.dec[6], f[6]);
    pull_row<S, SHIFTED, V, -1, HINT>(pn + 7 * plane, lane, x0, pitch, C(1.0 / 36.0), q.dec[7], f[7]);
    pull_row<S, SHIFTED, V, 1, HINT>(pn + 8 * plane, lane, x0, pitch, C(1.0 / 36.0), q.dec[8], f[8]);
    if (x0 == 0)
#pragma unroll
        for (int j = 0; j < 9; ++j) f[j][0] = f[j][V > 1 ? 1 : 0];
    const int sR = nx - 1 - x0;  // slot of the right wall node in this lane, if any
#pragma unroll
    for (int i = 1; i < V; ++i)
        if (sR == i) {
#pragma unroll
            for (int j = 0; j < 9; ++j) f[j][i] = f[j][i - 1];
        }
    if (sR == 0) {  // x_f = nx - 2 belongs to the previous lane: pull it directly
        const long long xf = nx - 2;
#pragma unroll
        for (int j = 0; j < 9; ++j) {
            const C v = ld1<S, HINT>(src + j * plane + (long long)(yc - cy(j)) * pitch + (xf - cx(j)), q.dec[j]);
            f[j][0] = SHIFTED ? v : v - C(wd(j));
        }
    }
}

// Observing points as the row step sees them: the up-to-four probes of a single cavity
// (kernel parameter space) or the one probe of a batched cavity (registers).
struct ProbeList {
    const ProbeSet& p;
    __device__ int n() const { return p.n; }
    __device__ int px(int q) const { return p.px[q]; }
    __device__ int py(int q) const { return p.py[q]; }
    __device__ int every(int q) const { return p.every[q]; }
    __device__ long long start(int q) const { return p.start[q]; }
    __device__ long long cap(int q) const { return p.cap[q]; }
    __device__ double* series(int q) const { return p.series[q]; }
};
struct ProbeOne {
    int n_, px_, py_, every_;
    long long start_, cap_;
    double* series_;
    __device__ int n() const { return n_; }
    __device__ int px(int) const { return px_; }
    __device__ int py(int) const { return py_; }
    __device__ int every(int) const { return every_; }
    __device__ long long start(int) const { return start_; }
    __device__ long long cap(int) const { return cap_; }
    __device__ double* series(int) const { return series_; }
};

// Geometry and parameters of one cavity as the row step sees them.
template <typename C>
struct CavityView {
    int nx, ny;
    long long pitch, plane;
    C omega, Ulid;
    int corner_moving;
    Relax<C> rx;     // FP64 only
    QCodec q;        // LBM_Q16S only
    C sref, sref_w;  // LBM_Q16S only: rho_ref the populations are read against / stored against
};

// One time step for the V nodes of lane `lane` in row y (x0 = first node): pull, moments,
// collision or wall closure, optional Eq. 6 accumulation and probe sampling, store.
// step_time() = global index of the step being produced (called only when a probe sits in this
// segment).
// EDGE_ALWAYS: run every warp through the node code with the wall tests instead of giving
// all-interior warps their own copy (the batch kernel's choice for 16-bit storage, below).
template <typename S, bool SHIFTED, bool REDUCE, int V, int HINT, bool EDGE_ALWAYS, typename Probes, typename TimeFn>
__device__ __forceinline__ void step_row(const S* __restrict__ src, S* __restrict__ dst,
                                         const CavityView<typename St<S>::C>& cv, int lane, int x0,
                                         int y, typename St<S>::C* snap, const Probes& probes,
                                         TimeFn step_time,
                                         typename St<S>::C& acc_drho, typename St<S>::C& acc_num,
                                         typename St<S>::C& acc_den) {
    using C = typename St<S>::C;
    const int nx = cv.nx, ny = cv.ny;
    const long long pitch = cv.pitch, plane = cv.plane;
    Relax<C> rx;
    if constexpr (sizeof(C) == 8) rx = cv.rx;
    else rx = make_relax<C>(cv.omega);
    const Omega<float> om = make_omega<float>(float(cv.omega));
    C f[9][V];
    pull_segment<S, SHIFTED, V, HINT>(src, lane, x0, y, nx, ny, pitch, plane, cv.q, f);
    // LBM_Q16S works on h = g - w rho_ref: BGK and the wall closure keep their form in h with
    // rho = 1 + rho_ref + sum h (sum w = 1, sum c w = 0); other storage types have rho_ref = 0
    const C one_ref = kIsQ16<S> ? C(1.0) + cv.sref : C(1.0);
    C sx[V], sy[V];
    if constexpr (REDUCE) {
        cload<C, V, HINT == 2>(snap + (long long)y * pitch + x0, sx);
        cload<C, V, HINT == 2>(snap + plane + (long long)y * pitch + x0, sy);
    }
    // observing points on this row segment (Sec. 3.3)
    unsigned pmask = 0;
    for (int q = 0; q < probes.n(); ++q)
        if (probes.py(q) == y && probes.px(q) >= x0 && probes.px(q) < x0 + V) pmask |= 1u << q;
    // Per node.  EDGE = false: every segment of the warp is interior (no wall, lid or padding
    // node), the case of all but the first and last warps of a row, so the wall tests compile
    // away; the arithmetic is the same either way.  The choice is made per warp (a per-lane choice
    // would run both copies of the node code in a warp that holds a wall lane).  With EDGE_ALWAYS
    // there is one copy: the batch kernel's 16-bit instantiations measured faster that way (half
    // the warps of a 500-wide cavity hold a wall lane; 45-cavity batch, f16s 131.4 -> 135.3 GLUPS),
    // while the single-cavity 16-bit kernel gains from the split (4096^2 f16s 171.4 -> 177.6).
    auto node = [&](auto edge_c, int i) {
        constexpr bool EDGE = decltype(edge_c)::value;
        const int x = x0 + i;
        C g[9];
#pragma unroll
        for (int j = 0; j < 9; ++j) g[j] = f[j][i];
        C out[9], drho, rho, ux, uy;
        constexpr bool PAIRS = kOnPairs<S, SHIFTED>;
        const bool wall = EDGE && ((y == 0) | (y == ny - 1) | (x == 0) | (x >= nx - 1));
        constexpr bool F64 = sizeof(C) == 8;
        C vel = C(1.0);
        if constexpr (F64) vel = wall ? rx.wall : rx.one;
        if constexpr (F64 && EDGE) collide<C, true>(g, one_ref, rx, out, drho, rho, ux, uy, vel);
        else if constexpr (PAIRS) collide<C>(g, one_ref, rx, out, drho, rho, ux, uy);
        else moments9(g, one_ref, drho, rho, ux, uy);
        C uox = ux, uoy = uy;
        if (wall) {
            const bool lid = (y == ny - 1) && (cv.corner_moving || (x > 0 && x < nx - 1));
            uox = lid ? cv.Ulid : C(0.0);
            uoy = C(0.0);
            if constexpr (F64) {
                if (lid) lid_shift<C>(rho, uox, out);
            } else if constexpr (PAIRS) wall_shift<C>(rho, ux, uy, uox, out);
            else if constexpr (kMomentum<S>) wall9(g, drho, rho, ux, uy, uox, cv.omega, out);
            else wall9_contracted(g, drho, rho, ux, uy, uox, cv.omega, out);
        } else if constexpr (!PAIRS) {
            collide9<kMomentum<S>>(g, drho, rho, ux, uy, om, out);
        }
#pragma unroll
        for (int j = 0; j < 9; ++j) f[j][i] = out[j];
        if (EDGE && x >= nx) {
#pragma unroll
            for (int j = 0; j < 9; ++j) f[j][i] = C(0.0);
        }
        if constexpr (REDUCE) {
            if (!EDGE || x < nx) {
                const C dx = uox - sx[i], dy = uoy - sy[i];  // exact when close (Sterbenz)
                acc_drho += kIsQ16<S> ? drho + cv.sref : drho;
                acc_num += dx * dx + dy * dy;
                acc_den += sx[i] * sx[i] + sy[i] * sy[i];
            }
            sx[i] = (!EDGE || x < nx) ? uox : C(0);
            sy[i] = (!EDGE || x < nx) ? uoy : C(0);
        }
        if (pmask) {
            for (int q = 0; q < probes.n(); ++q) {
                if (((pmask >> q) & 1u) && probes.px(q) == x) {
                    const long long t = step_time();
                    const int ev = probes.every(q);
                    if (t % ev == 0) {
                        long long k = t / ev - probes.start(q) / ev - 1;
                        if (k >= 0) {
                            k %= probes.cap(q);
                            probes.series(q)[2 * k] = double(uox);
                            probes.series(q)[2 * k + 1] = double(uoy);
                        }
                    }
                }
            }
        }
    };
    if (EDGE_ALWAYS || __any_sync(kFull, (y == 0) | (y == ny - 1) | (x0 == 0) | (x0 + V >= nx))) {
#pragma unroll
        for (int i = 0; i < V; ++i) node(std::true_type{}, i);
    } else {
#pragma unroll
        for (int i = 0; i < V; ++i) node(std::false_type{}, i);
    }

    S* pd = dst + (long long)y * pitch + x0;
    bool sat = false;
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        if constexpr (!SHIFTED) {
#pragma unroll
            for (int i = 0; i < V; ++i) f[j][i] += C(wd(j));
        }
        if constexpr (kIsQ16<S> && REDUCE) {  // re-reference to the next rho_ref
            const C shift = C(wd(j)) * (cv.sref - cv.sref_w);
#pragma unroll
            for (int i = 0; i < V; ++i)
                if (x0 + i < nx) f[j][i] += shift;
        }
        vstore_g<S, V>(pd + j * plane, cv.q.enc[j], f[j], sat);
    }
    if constexpr (kIsQ16<S> && REDUCE) {
        if (sat) acc_num += C(NAN);  // a saturated code: the checkpoint reports non-finite
    }
    if constexpr (REDUCE) {
        cstore<C, V>(snap + (long long)y * pitch + x0, sx);
        cstore<C, V>(snap + plane + (long long)y * pitch + x0, sy);
    }
}

// Sum of three per-thread values over the block's warps into partials[3*block .. 3*block+2].
template <int BY, typename C>
__device__ __forceinline__ void block_partials(C a0, C a1, C a2, double* partials, long long block) {
    __shared__ double red[3][BY];
    const double s0 = warp_sum(double(a0));
    const double s1 = warp_sum(double(a1));
    const double s2 = warp_sum(double(a2));
    if (threadIdx.x == 0) {
        red[0][threadIdx.y] = s0;
        red[1][threadIdx.y] = s1;
        red[2][threadIdx.y] = s2;
    }
    __syncthreads();
    if (threadIdx.y == 0 && threadIdx.x < 3) {
        double s = 0.0;
#pragma unroll
        for (int w = 0; w < BY; ++w) s += red[threadIdx.x][w];
        partials[3 * block + threadIdx.x] = s;
    }
}

// Resident blocks per SM the register budget is sized for.  binary16 / bfloat16 storage: 32 warps
// per SM (64 registers, a few spilled to L1).  Left to itself the compiler takes 80 and leaves 24
// warps, and these kernels wait on memory latency: f16s 163 -> 170 GLUPS at 4096^2 (bf16s 161 ->
// 168).  0 (no bound) for the rest -- a bound of 1 is not the same as none, it lets the compiler
// take more registers; LBM_Q16S, bound by its integer code conversions, lost 4 % at 2048^2 under
// the same cap.
template <typename S, int BY>
inline constexpr int kStepMinBlocks = (sizeof(S) == 2 && !kIsQ16<S>) ? 32 / BY : 0;

template <typename S, bool SHIFTED, bool REDUCE, int V, int R, int BY, int HINT>
__global__ void __launch_bounds__(32 * BY, (kStepMinBlocks<S, BY>)) k_step(const StepArgs a) {
    using C = typename St<S>::C;
    const int lane = threadIdx.x;
    const int x0 = (blockIdx.x * 32 + lane) * V;
    const int yb = (blockIdx.y * BY + threadIdx.y) * R;
    CavityView<C> cv;
    cv.nx = a.nx;
    cv.ny = a.ny;
    cv.pitch = a.pitch;
    cv.plane = a.plane;
    cv.omega = sizeof(C) == 4 ? C(a.omega_f) : C(a.omega);
    cv.Ulid = sizeof(C) == 4 ? C(a.U_f) : C(a.U);
    cv.corner_moving = a.corner_moving;
    if constexpr (sizeof(C) == 8) cv.rx = in_registers(a.rx);
    cv.sref = cv.sref_w = C(0);
    if constexpr (kIsQ16<S>) {
        cv.q = a.q;
        cv.sref = C(__ldcg(&a.state->rho_ref[0]));
        cv.sref_w = REDUCE ? C(__ldcg(&a.state->rho_ref[1])) : cv.sref;
    }
    const S* __restrict__ src = static_cast<const S*>(a.src);
    S* __restrict__ dst = static_cast<S*>(a.dst);
    C acc_drho = C(0), acc_num = C(0), acc_den = C(0);
#pragma unroll 1
    for (int r = 0; r < R; ++r) {
        const int y = yb + r;
        if (y >= a.ny) break;  // uniform across the warp
        step_row<S, SHIFTED, REDUCE, V, HINT, kIsQ16<S>>(
            src, dst, cv, lane, x0, y, static_cast<C*>(a.snap), ProbeList{a.probes},
            [&]() { return a.state->base + a.s + 1; }, acc_drho, acc_num, acc_den);
    }
    if constexpr (REDUCE) block_partials<BY>(acc_drho, acc_num, acc_den, a.partials, (long long)blockIdx.y * gridDim.x + blockIdx.x);
}

// Launch shape (nodes per lane V, rows per thread R, warps per block BY, load hint).  Every shape
// computes bitwise-identical populations; only speed differs.
template <typename S, bool SHIFTED, int V, int R, int BY, int HINT>
static cudaError_t launch_step_shape(const StepArgs& a, bool reduce, cudaStream_t st) {
    dim3 block(32, BY);
    dim3 grid((unsigned)((a.nx + 32 * V - 1) / (32 * V)), (unsigned)((a.ny + BY * R - 1) / (BY * R)));
    if (reduce)
        k_step<S, SHIFTED, true, V, R, BY, HINT><<<grid, block, 0, st>>>(a);
    else
        k_step<S, SHIFTED, false, V, R, BY, HINT><<<grid, block, 0, st>>>(a);
    return cudaGetLastError();
}

// The shape tables; kShapes* in lbm_step.cu mirror them.
template <typename S, bool SHIFTED>
static cudaError_t launch_step_cfg(int cfg, const StepArgs& a, bool reduce, cudaStream_t st) {
    // nodes per lane: 1 for FP64 (default_step_config), 2 for FP32 storage (8-byte vectors; the smaller
    // register footprint buys more resident warps, measured faster than 4), 4 for 16-bit storage; 1 in
    // the FP32 shape for small grids, which spreads the nodes over as many warps as there are
    if constexpr (sizeof(S) == 8) {
        switch (cfg) {
            case 0: return launch_step_shape<S, SHIFTED, 1, 2, 2, 0>(a, reduce, st);
            case 1: return launch_step_shape<S, SHIFTED, 1, 2, 4, 0>(a, reduce, st);
            case 2: return launch_step_shape<S, SHIFTED, 1, 1, 4, 0>(a, reduce, st);
            case 3: return launch_step_shape<S, SHIFTED, 1, 4, 1, 0>(a, reduce, st);
            case 4: return launch_step_shape<S, SHIFTED, 1, 2, 1, 0>(a, reduce, st);
            case 5: return launch_step_shape<S, SHIFTED, 1, 1, 1, 0>(a, reduce, st);
            default: return cudaErrorInvalidValue;
        }
    } else {
        constexpr int V = sizeof(S) == 2 ? 4 : 2;
        constexpr bool WIDE = sizeof(S) == 4;
        switch (cfg) {
            case 0: return launch_step_shape<S, SHIFTED, V, 2, 2, 0>(a, reduce, st);
            case 1: return launch_step_shape<S, SHIFTED, V, 1, 4, 0>(a, reduce, st);
            case 2: return launch_step_shape<S, SHIFTED, WIDE ? 1 : V, WIDE ? 1 : 2, WIDE ? 4 : 2, WIDE ? 0 : 1>(a, reduce, st);
            case 3: return launch_step_shape<S, SHIFTED, V, 4, 1, 0>(a, reduce, st);
            case 4: return launch_step_shape<S, SHIFTED, V, 2, 4, 0>(a, reduce, st);
            case 5: return launch_step_shape<S, SHIFTED, V, WIDE ? 2 : 4, 2, 1>(a, reduce, st);
            default: return cudaErrorInvalidValue;
        }
    }
}

}  // namespace lbm
