// Device code of the D3Q27 central-Hermite MRT step (included once per
// storage precision by step_fp64.cu / step_fp32.cu / step_fp16s.cu).
//
// Method (arXiv 2204.10566):
//   f_i(x + c_i, t + 1) = f_i + [T^-1 S T (f^eq - f)]_i           (Sec. 2.1)
//   T_{m,i} = H_m(c_i - u): central Hermite moments                 (Sec. 2.1)
//   f^eq: full Hermite expansion on D3Q27 (Appendix A), whose central
//   moments are (rho, 0, ..., 0)                                    (Appendix A)
//   second-order moments relaxed at omega, orders 3..6 at the ghost rates
//   (default 1, Appendix A).
//
// GB300 design: pull scheme over a fluid-only slot layout (rows of cells
// contiguous along the lattice's longer axis), structure-of-arrays
// populations stored as deviations from the lattice weights; one warp per
// tile of up to 32 cells of a row (FP32), one thread per two cells over staged
// copies (FP16S, larger lattices) or one thread per cell (smaller FP16S,
// FP64), with the inlet/outlet nodes and the interpolated-wall cells in
// kernels of their own on a second stream.  Every pull source has a
// slot (wall links read a ghost slot the cell filled with its reflected
// population in the previous step), so the gather is 27 unconditional
// coalesced loads at nb[j] + x - cx.  Because T(u) is the tensor product of
// three 1-D 3x3 transforms, T and its inverse are applied as a cascade of
// 1-D passes in registers; with the default ghost rates only the six
// second-order central moments survive relaxation and the inverse is the
// product-form equilibrium plus six correction terms.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "lbm_internal.h"

// Minimum resident blocks per SM requested for the FP32 / FP16S step kernel
// (caps its registers: 65536 / (threads * blocks)); FP64 is left uncapped.
#ifndef LBM_STEP_MIN_BLOCKS
#define LBM_STEP_MIN_BLOCKS 8
#endif
// When the FP32 chunk kernel runs (LBM_FLUID_KERNEL=chunk), the inlet/outlet
// nodes ride in its trailing blocks instead of a launch of their own: +2 % on
// the Re 3500 nozzle, although the node path spills at the fluid path's
// register cap.  In FP16S the fused kernel spilled in the fluid path too, and
// FP64's uncapped fluid path would lose occupancy, so both keep the separate
// launch.
// FP16S: gather and own-slot stores addressed from one pointer per line
// (the three values of a line sit at +1, +stride, +2 stride - 1 from it):
// +4 % / +7 % on the Re 3500 / Re 6500 nozzles, while FP32 lost 4 %, so FP32
// keeps per-population offsets.
#ifndef LBM_LINE_POINTERS
#define LBM_LINE_POINTERS 1
#endif
#ifndef LBM_FUSE_BOUNDARY
#define LBM_FUSE_BOUNDARY 1
#endif
// Warp-uniform fast path of the FP32 / FP16S fluid kernel for warps of fluid
// cells without wall links (fluid_lane_voted); 0 runs every warp through the
// general line sink.
#ifndef LBM_FAST_PATH
#define LBM_FAST_PATH 1
#endif
// Minimum resident blocks of the kernel of the cells with interpolated walls,
// which keeps the wall record and the own-slot values of a cell in registers as
// well.
#ifndef LBM_STEP_MIN_BLOCKS_WALLQ
#define LBM_STEP_MIN_BLOCKS_WALLQ 4
#endif
// L2 prefetch lookahead of the fluid kernel, in percent of the blocks
// resident on the device (0 disables the prefetch).  At 8 blocks per SM the
// FP32 kernel keeps enough loads in flight on its own (the prefetch measured
// neutral, +60 MB of DRAM reads per Re 3500 step), and FP16S runs 2-3 %
// slower with it; both default to off.
#ifndef LBM_PREFETCH_AHEAD_PCT
#define LBM_PREFETCH_AHEAD_PCT 0
#endif
#ifndef LBM_PREFETCH_AHEAD_PCT_FP16S
#define LBM_PREFETCH_AHEAD_PCT_FP16S 0
#endif


namespace lbm {

// ------------------------------------------------------------- storage types

// A population load: through the read-only path, or (CG) from L2, for a
// kernel that also writes the array in another step.
template <bool CG, class T>
__device__ __forceinline__ T fetch(const T *p) {
    if constexpr (CG)
        return __ldcg(p);
    else
        return __ldg(p);
}

template <int P>
struct Storage;

template <>
struct Storage<0> {  // FP64 deviations
    using T = double;
    using R = double;
    template <bool CG = false>
    static __device__ __forceinline__ R load(const T *p, R) { return fetch<CG>(p); }
    template <bool CG = false>
    static __device__ __forceinline__ R load_raw(const T *p) { return fetch<CG>(p); }
    static __device__ __forceinline__ void store_raw(T *p, R v) { *p = v; }
    static constexpr bool SCALED = false;
    static __device__ __forceinline__ void store(T *p, R v, R) { *p = v; }
};

template <>
struct Storage<1> {  // FP32 deviations
    using T = float;
    using R = float;
    template <bool CG = false>
    static __device__ __forceinline__ R load(const T *p, R) { return fetch<CG>(p); }
    template <bool CG = false>
    static __device__ __forceinline__ R load_raw(const T *p) { return fetch<CG>(p); }
    static __device__ __forceinline__ void store_raw(T *p, R v) { *p = v; }
    static constexpr bool SCALED = false;
    static __device__ __forceinline__ void store(T *p, R v, R) { *p = v; }
};

template <>
struct Storage<2> {  // FP16 (f - w) * s, FP32 arithmetic
    using T = __half;
    using R = float;
    template <bool CG = false>
    static __device__ __forceinline__ R load(const T *p, R inv_s) { return __half2float(fetch<CG>(p)) * inv_s; }
    template <bool CG = false>
    static __device__ __forceinline__ R load_raw(const T *p) { return __half2float(fetch<CG>(p)); }
    static __device__ __forceinline__ void store_raw(T *p, R v) { *p = __float2half_rn(v); }
    static constexpr bool SCALED = true;
    static __device__ __forceinline__ void store(T *p, R v, R s) { *p = __float2half_rn(v * s); }
};

// ----------------------------------------------------------------- stencil

__host__ __device__ constexpr int cx_of(int i) { return i % 3 - 1; }
__host__ __device__ constexpr int cy_of(int i) { return (i / 3) % 3 - 1; }
__host__ __device__ constexpr int cz_of(int i) { return i / 9 - 1; }

// Storage addressing of a lattice whose rows run along axis AX (0: x, 2: z):
// the pull source of population i of the cell at row position p is slot
// nb[row_line<AX>(i)] + p - c_row<AX>(i).
template <int AX>
__host__ __device__ constexpr int c_row(int i) { return AX == 0 ? cx_of(i) : cz_of(i); }
template <int AX>
__host__ __device__ constexpr int row_line(int i) { return AX == 0 ? i / 3 : (cx_of(i) + 1) + 3 * (cy_of(i) + 1); }
// Population of storage line j with c_row = k - 1 (k = 0, 1, 2).
template <int AX>
__host__ __device__ constexpr int line_pop(int j, int k) { return AX == 0 ? 3 * j + k : j + 9 * k; }

// 1-D Gauss-Hermite weights of the third-order quadrature (Appendix A).
// Scalar type of R (F2 holds two FP32 values).
template <class R>
struct ScalarOf {
    using type = R;
};
template <>
struct ScalarOf<struct F2> {
    using type = float;
};

template <class R>
__device__ __forceinline__ R w1(int c) {
    using X = typename ScalarOf<R>::type;
    return R(c == 0 ? X(2) / X(3) : X(1) / X(6));
}

template <class R>
__device__ __forceinline__ R theta0() {
    using X = typename ScalarOf<R>::type;
    return R(X(1) / X(3));
}

// The rational constant a / b in the scalar precision of R.
template <class R>
__device__ __forceinline__ R cst(int a, int b) {
    using X = typename ScalarOf<R>::type;
    return R(X(a) / X(b));
}

// 1-D inverse-transform columns at velocity u (T_1D(u)^-1, column k = g_k):
//   g0(c) = w(c) + d(c), d(0) = -u^2, d(+-1) = (u^2 +- u)/2
//   g1(0) = -2u, g1(+-1) = u +- 1/2;  g2(0) = -1, g2(+-1) = 1/2.
// g0 is also the 1-D factor of the product-form equilibrium.
template <class R>
struct Axis {
    R d[3], g0[3], g1[3];
    // lo, hi: u^2 - u and u^2 + u in one rounding each, else the square is rounded first
    __device__ __forceinline__ Axis(R u, bool lo, bool hi);
};

template <class R>
__device__ __forceinline__ R g2(int c) { return c == 0 ? R(-1) : R(0.5); }

// Arithmetic with the rounding written out (no contraction by the compiler),
// so that one cell per thread (float) and two cells per thread (F2) round
// alike whatever kernel the code is inlined into.
__device__ __forceinline__ float fma_(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float add_(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub_(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float mul_(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double add_(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub_(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double mul_(double a, double b) { return __dmul_rn(a, b); }

// ------------------------------------------------------ viscous stress

// Viscous stress of a cell from its pre-collision second-order central
// Hermite moments a_ab = sum_i ((c - u)_a (c - u)_b - theta0 delta_ab) f_i
// (Appendix A strain-rate relation, with the sign of the non-equilibrium
// stress): sigma_ab = 2 rho nu S_ab = -(1 - omega/2) a_ab, accumulated in
// FP64 on statistics sample steps (Sec. 2.2 viscous shear stress).
template <class R>
__device__ __forceinline__ void record_stress(const StepArgs &a, int slot, R omega, const R (&a2)[6]) {
    if ((a.flags & (STEP_STATS | STEP_STATS_FULL)) != (STEP_STATS | STEP_STATS_FULL)) return;
    const double f = -(1.0 - 0.5 * (double)omega);
    double *p = a.stats + 11 * (int64_t)a.stride + slot;
#pragma unroll
    for (int q = 0; q < 6; ++q) p[q * a.stride] = fma_(f, (double)a2[q], p[q * a.stride]);
}

// --------------------------------------------------------------- collision

__device__ __forceinline__ float recip(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double recip(double x) { return 1.0 / x; }

__device__ __forceinline__ float2 bc2(float a) { return make_float2(a, a); }

// Two cells' FP32 values on the packed pipe: every arithmetic operation of
// the collision applies to both lanes with one instruction.
struct F2 {
    float2 v;
    F2() = default;
    __device__ __forceinline__ F2(float s) : v(make_float2(s, s)) {}
    __device__ __forceinline__ explicit F2(float2 w) : v(w) {}
};
__device__ __forceinline__ F2 operator+(F2 a, F2 b) { return F2(__fadd2_rn(a.v, b.v)); }
__device__ __forceinline__ F2 operator-(F2 a, F2 b) { return F2(__ffma2_rn(b.v, bc2(-1.0f), a.v)); }
__device__ __forceinline__ F2 operator-(F2 a) { return F2(__fmul2_rn(a.v, bc2(-1.0f))); }
__device__ __forceinline__ F2 operator*(F2 a, F2 b) { return F2(__fmul2_rn(a.v, b.v)); }
__device__ __forceinline__ F2 &operator+=(F2 &a, F2 b) { return a = a + b; }
__device__ __forceinline__ F2 &operator*=(F2 &a, F2 b) { return a = a * b; }
__device__ __forceinline__ F2 recip(F2 x) { return F2(make_float2(__frcp_rn(x.v.x), __frcp_rn(x.v.y))); }

// The same on two cells at once.
__device__ __forceinline__ F2 fma_(F2 a, F2 b, F2 c) { return F2(__ffma2_rn(a.v, b.v, c.v)); }
__device__ __forceinline__ F2 add_(F2 a, F2 b) { return a + b; }
__device__ __forceinline__ F2 sub_(F2 a, F2 b) { return a - b; }
__device__ __forceinline__ F2 mul_(F2 a, F2 b) { return a * b; }
// Sums with a product that was rounded on its own: cell by cell, since the
// compiler takes a packed product and a packed sum together (and a packed
// multiply-add by one as a sum).
__device__ __forceinline__ F2 add_apart(F2 a, F2 b) { return F2(make_float2(__fadd_rn(a.v.x, b.v.x), __fadd_rn(a.v.y, b.v.y))); }
__device__ __forceinline__ float add_apart(float a, float b) { return __fadd_rn(a, b); }

template <class R>
__device__ __forceinline__ R pick(bool a, R x, R y) { return a ? x : y; }
template <>
__device__ __forceinline__ F2 pick(bool a, F2 x, F2 y) { return F2(make_float2(a ? x.v.x : y.v.x, a ? x.v.y : y.v.y)); }

template <class R>
__device__ __forceinline__ Axis<R>::Axis(R u, bool lo, bool hi) {
    const R h = R(0.5), u2 = mul_(u, u);
    const R m = pick(lo, fma_(u, u, -u), add_apart(u2, -u)), p = pick(hi, fma_(u, u, u), add_apart(u2, u));
    d[0] = mul_(h, m);
    d[1] = -u2;
    d[2] = mul_(h, p);
    g0[0] = fma_(h, m, w1<R>(-1));
    g0[1] = sub_(w1<R>(0), u2);
    g0[2] = fma_(h, p, w1<R>(1));
    g1[0] = sub_(u, h);
    g1[1] = mul_(R(-2), u);
    g1[2] = add_(u, h);
}

// Shared inputs of the per-line inverse (see collide_ghost1).
template <class R>
struct PairCoef {
    R Axx, Ayy, Azz, Axy, Axz, Ayz, rho_o, drho_o, ux, ux2h, uxh;
};

// Line (cy, cz) = (0, 0) of the inverse: f*_i - w_i for cx = -1, 0, +1.
template <class R, class Out>
__device__ __forceinline__ void inverse_centre(const PairCoef<R> &c, const Axis<R> &Y, const Axis<R> &Z,
                                               const Out &sink) {
    const R h = R(0.5f), w0 = cst<R>(2, 3), w1_ = cst<R>(1, 6), w00 = R(cst<float>(2, 3) * cst<float>(2, 3));
    const R gy0 = Y.g0[1], gz0 = Z.g0[1], gy1 = Y.g1[1], gz1 = Z.g1[1];
    const R E = mul_(gy0, gz0);
    const R D = fma_(w0, Z.d[1], mul_(Y.d[1], gz0));
    const R C0 = fma_(mul_(c.Ayz, gy1), gz1, fma_(-c.Azz, gy0, mul_(-c.Ayy, gz0)));
    const R B1 = fma_(mul_(c.Axy, gy1), gz0, mul_(mul_(c.Axz, gy0), gz1));
    const R B2 = mul_(c.Axx, E);
    const R Bw = add_(fma_(c.drho_o, w00, mul_(c.rho_o, D)), C0);
    const R Bd = fma_(c.rho_o, E, C0), xBd = mul_(c.ux2h, Bd);
    const R v0 = sub_(fma_(w0, Bw, mul_(R(-2.0f), fma_(c.ux, B1, xBd))), B2);
    const R S = fma_(h, B2, fma_(c.ux, B1, fma_(w1_, Bw, xBd)));
    const R A = fma_(h, B1, mul_(c.uxh, Bd));
    sink(4, sub_(S, A), v0, add_(S, A));
}

// Two lines of the inverse at once.  The pair differs along one axis ("v",
// c = -1 in .x and +1 in .y) and shares the other ("f"); the line formulas
// are symmetric in y and z once the diagonal and mixed second-order
// coefficients are relabelled, so one routine serves both kinds of pair:
//   E = g0v g0f,  D = dv g0f + (1/6) df,
//   C0 = Avv (1/2) g0f + Aff g2f g0v + Ayz g1f g1v,
//   B1 = Axv g0f g1v + Axf g1f g0v,  B2 = Axx E,
// with the same Bw, Bd, v0, S, A as the scalar line.
template <int JA, int JB, class Out>
__device__ __forceinline__ void inverse_pair(const PairCoef<float> &c, const Axis<float> &Y, const Axis<float> &Z,
                                             const Out &sink) {
    constexpr bool YV = (JA / 3) == (JB / 3);  // same cz: y varies
    constexpr int cf = YV ? JA / 3 - 1 : JA % 3 - 1;  // fixed axis velocity
    const Axis<float> &V = YV ? Y : Z;
    const Axis<float> &F = YV ? Z : Y;
    const float Avv = YV ? c.Ayy : c.Azz, Aff = YV ? c.Azz : c.Ayy;
    const float Axv = YV ? c.Axy : c.Axz, Axf = YV ? c.Axz : c.Axy;
    const float f0 = F.g0[cf + 1], f1 = F.g1[cf + 1], fd = F.d[cf + 1], fw = w1<float>(cf), fg2 = g2<float>(cf);
    const float2 v0_ = make_float2(V.g0[0], V.g0[2]), v1_ = make_float2(V.g1[0], V.g1[2]);
    const float2 vd = make_float2(V.d[0], V.d[2]);
    const float2 E = __fmul2_rn(v0_, bc2(f0));
    const float2 D = __ffma2_rn(vd, bc2(f0), bc2(mul_(fd, 1.0f / 6.0f)));
    const float2 C0 = __ffma2_rn(v1_, bc2(mul_(c.Ayz, f1)), __ffma2_rn(v0_, bc2(mul_(Aff, fg2)), bc2(mul_(mul_(0.5f, Avv), f0))));
    const float2 hB1 = __ffma2_rn(v1_, bc2(mul_(mul_(0.5f, Axv), f0)), __fmul2_rn(v0_, bc2(mul_(mul_(0.5f, Axf), f1))));
    const float2 nB2 = __fmul2_rn(v0_, bc2(mul_(-c.Axx, f0)));
    const float2 Bw = __ffma2_rn(bc2(c.rho_o), D, __fadd2_rn(C0, bc2(mul_(c.drho_o, fw * (1.0f / 6.0f)))));
    const float2 Bd = __ffma2_rn(bc2(c.rho_o), E, C0);
    const float2 t = __ffma2_rn(bc2(c.ux2h), Bd, __fmul2_rn(bc2(mul_(2.0f, c.ux)), hB1));
    const float2 o0 = __ffma2_rn(bc2(2.0f / 3.0f), Bw, __ffma2_rn(bc2(-2.0f), t, nB2));
    const float2 S = __ffma2_rn(bc2(1.0f / 6.0f), Bw, __ffma2_rn(v0_, bc2(mul_(mul_(0.5f, c.Axx), f0)), t));
    const float2 A = __ffma2_rn(bc2(c.uxh), Bd, hB1);
    const float2 om = __ffma2_rn(bc2(-1.0f), A, S), op = __fadd2_rn(S, A);
    sink(JA, om.x, o0.x, op.x);
    sink(JB, om.y, o0.y, op.y);
}

// inverse_pair for two cells, a cell to a packed lane: one line after the
// other, each value in the same order of operations.
template <int JA, int JB, class Out>
__device__ __forceinline__ void inverse_pair(const PairCoef<F2> &c, const Axis<F2> &Y, const Axis<F2> &Z,
                                             const Out &sink) {
    constexpr bool YV = (JA / 3) == (JB / 3);
    constexpr int cf = YV ? JA / 3 - 1 : JA % 3 - 1;
    const Axis<F2> &V = YV ? Y : Z;
    const Axis<F2> &F = YV ? Z : Y;
    const F2 Avv = YV ? c.Ayy : c.Azz, Aff = YV ? c.Azz : c.Ayy;
    const F2 Axv = YV ? c.Axy : c.Axz, Axf = YV ? c.Axz : c.Axy;
    const F2 h = F2(0.5f), f0 = F.g0[cf + 1], f1 = F.g1[cf + 1], fd = mul_(F.d[cf + 1], F2(1.0f / 6.0f));
    const F2 P = mul_(c.Ayz, f1), Q = mul_(Aff, g2<F2>(cf)), C = mul_(mul_(h, Avv), f0);
    const F2 b1 = mul_(mul_(h, Axv), f0), b0 = mul_(mul_(h, Axf), f1), x0 = mul_(mul_(h, c.Axx), f0), n0 = mul_(-c.Axx, f0);
    const F2 w = mul_(c.drho_o, F2(w1<float>(cf) * (1.0f / 6.0f))), u2 = mul_(F2(2.0f), c.ux);
#pragma unroll
    for (int k = 0; k < 3; k += 2) {
        const F2 v0 = V.g0[k], v1 = V.g1[k];
        const F2 E = mul_(v0, f0), D = fma_(V.d[k], f0, fd), C0 = fma_(v1, P, fma_(v0, Q, C)), hB1 = fma_(v1, b1, mul_(v0, b0));
        const F2 Bw = fma_(c.rho_o, D, add_apart(C0, w)), Bd = fma_(c.rho_o, E, C0);
        const F2 t = fma_(c.ux2h, Bd, mul_(u2, hB1)), A = fma_(c.uxh, Bd, hB1);
        const F2 o0 = fma_(F2(2.0f / 3.0f), Bw, fma_(F2(-2.0f), t, mul_(v0, n0)));
        const F2 S = fma_(F2(1.0f / 6.0f), Bw, fma_(v0, x0, t));
        sink(k ? JB : JA, sub_(S, A), o0, add_(S, A));
    }
}

// Writes a line of three outputs (cx = -1, 0, +1 of line j) back into d.
template <class R>
struct ToArray {
    R (&d)[27];
    __device__ __forceinline__ void moments(R, const R (&)[6]) const {}
    __device__ __forceinline__ void operator()(int j, R vm, R v0, R vp) const {
        d[3 * j] = vm;
        d[3 * j + 1] = v0;
        d[3 * j + 2] = vp;
    }
};

// ToArray that also records the viscous stress of the cell at `slot`.
template <class R>
struct ToArrayStress {
    const StepArgs &a;
    int slot;
    R (&d)[27];
    __device__ __forceinline__ void moments(R omega, const R (&a2)[6]) const { record_stress(a, slot, omega, a2); }
    __device__ __forceinline__ void operator()(int j, R vm, R v0, R vp) const { ToArray<R>{d}(j, vm, v0, vp); }
};

// Moment sums of the FP32 and FP16S collisions: m = drho, jx, jy, jz, pxx,
// pyy, pzz, pxy, pxz, pyz, the sums of (f - w) weighted by 1, c, and c_a c_b;
// ld(i) gives f_i - w_i, or a power of two times it, of one cell (R = float)
// or two (R = F2).  The x-pass sums each (cy, cz) line with weights 1, cx,
// cx^2; the other axes follow.
template <class R, class Load>
__device__ __forceinline__ void ghost1_sums(const Load &ld, R (&m)[10]) {
    R s0[9], s1[9], s2[9];
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        const R a = ld(3 * j), b = ld(3 * j + 1), c = ld(3 * j + 2);
        s0[j] = (a + b) + c;
        s1[j] = c - a;
        s2[j] = c + a;
    }
    R drho = s0[0], jx = s1[0], pxx = s2[0];
#pragma unroll
    for (int j = 1; j < 9; ++j) {
        drho += s0[j];
        jx += s1[j];
        pxx += s2[j];
    }
    // lines in storage order, each pair of a column's first two at once
    const R jy = (((((s0[2] - s0[0]) - s0[3]) + s0[5]) - s0[6]) + s0[8]), pyy = ((((s0[0] + s0[2]) + s0[3]) + s0[5]) + s0[6]) + s0[8];
    const R pxy = ((((s1[2] - s1[0]) - s1[3]) + s1[5]) - s1[6]) + s1[8];
    // z: lines 0 1 2 against 6 7 8, one after the other
    const R zn = (s0[0] + s0[1]) + s0[2], xn = (s1[0] + s1[1]) + s1[2];
    const R jz = ((s0[6] - zn) + s0[7]) + s0[8], pzz = ((zn + s0[6]) + s0[7]) + s0[8], pxz = ((s1[6] - xn) + s1[7]) + s1[8];
    const R pyz = ((s0[0] - s0[2]) - s0[6]) + s0[8];
    m[0] = drho, m[1] = jx, m[2] = jy, m[3] = jz, m[4] = pxx;
    m[5] = pyy, m[6] = pzz, m[7] = pxy, m[8] = pxz, m[9] = pyz;
}

// Roundings of the rate-1 collision in FP32 arithmetic.  Where a product
// meets a sum it is rounded before the sum or taken into it (a fused
// multiply-add), and FP16 storage carries such a difference on: in some 50
// steps it grows to the size of the storage's own noise, 1e-3 of a velocity.
// So each FP16S cell keeps one set of roundings whatever kernel updates it and
// whether statistics are sampled: whole warps of plain cells in the chunk list
// (CHUNK_PLAIN) and cells with interpolated walls take the default, the other
// cells lane_rounds, the request server's served_rounds.  y, z: u_y^2 -+ u_y
// and u_z^2 + u_z in one rounding; late: the second-order moments' scale first.
struct Rounds {
    bool y = false, z = false, late = false;
};
template <int AX>
__device__ __forceinline__ Rounds lane_rounds(bool plain) { return {!plain, !plain && AX == 2, false}; }
__device__ __forceinline__ constexpr Rounds served_rounds() { return {true, true, true}; }

// The rest of the FP32 / FP16S default-rate collision from the moment sums:
// rho, u, the six second-order central Hermite moments, their relaxation, and
// the inverse transform, line by line into sink(j, f*_{3j} - w, f*_{3j+1} - w,
// f*_{3j+2} - w).  With SCALED (FP16S) the sums are of (f - w) / in_scale and
// the outputs are (f* - w) * out_scale: the scales, powers of two, act on the
// ten moments and the eight output coefficients.
template <bool SCALED, class R, class Out>
__device__ __forceinline__ void ghost1_finish(const R (&m)[10], R omega, R &rho, R &ux, R &uy, R &uz, R in_scale,
                                              R out_scale, Rounds rounds, const Out &sink) {
    const R drho = SCALED ? mul_(m[0], in_scale) : m[0], th = theta0<R>();
    rho = add_(R(1.0f), drho);
    const R inv = recip(rho);
    ux = mul_(SCALED ? mul_(m[1], in_scale) : m[1], inv);
    uy = mul_(SCALED ? mul_(m[2], in_scale) : m[2], inv);
    uz = mul_(SCALED ? mul_(m[3], in_scale) : m[3], inv);
    // Second-order central Hermite moments sum_i ((c-u)_a (c-u)_b - theta0 delta_ab) f_i,
    // from the deviation moments (sum c_a c_b w = theta0 delta_ab).
    const R rx = -mul_(rho, ux), ry = -mul_(rho, uy), rz = -mul_(rho, uz);
    auto less = [&](R p, R r, R u) {
        if (!SCALED) return fma_(r, u, p);
        return rounds.late ? fma_(r, u, mul_(p, in_scale)) : fma_(p, in_scale, mul_(r, u));
    };
    const R a2[6] = {fma_(-th, drho, less(m[4], rx, ux)), fma_(-th, drho, less(m[5], ry, uy)),
                     fma_(-th, drho, less(m[6], rz, uz)), less(m[7], rx, uy),
                     less(m[8], rx, uz),                  less(m[9], ry, uz)};
    sink.moments(omega, a2);
    // Inverse: f* = rho prod g0 + sum over the six relaxed second-order moments
    // of A_m prod_a g_{m_a}; orders 1 and 3..6 are zero after relaxation.
    // Per (cy, cz) line the x-dependence is spanned by {w, d, g1, g2}(cx):
    //   f*_i - w_i = wx Bw + dx Bd + g1x B1 + g2x B2,
    // and for cx = +-1 this splits into S +- A.  One cell's lines go in pairs
    // on the packed FP32 pipe (two lanes per instruction): (cy = -1, +1) at
    // each cz, then (cz = -1, +1) at cy = 0; two cells' lines one by one with a
    // cell to a lane; the centre line alone.
    const R one_w = sub_(R(1.0f), omega), k = SCALED ? mul_(one_w, out_scale) : one_w, uxh = mul_(R(0.5f), ux);
    const Axis<R> Y(uy, rounds.y, rounds.y), Z(uz, false, rounds.z);
    const PairCoef<R> c{mul_(k, a2[0]), mul_(k, a2[1]), mul_(k, a2[2]), mul_(k, a2[3]), mul_(k, a2[4]), mul_(k, a2[5]),
                        SCALED ? mul_(rho, out_scale) : rho, SCALED ? mul_(drho, out_scale) : drho, ux, mul_(uxh, ux), uxh};
    if constexpr (std::is_same<R, float>::value) {
        inverse_pair<0, 2>(c, Y, Z, sink);
        inverse_pair<3, 5>(c, Y, Z, sink);
        inverse_pair<6, 8>(c, Y, Z, sink);
        inverse_pair<1, 7>(c, Y, Z, sink);
        inverse_centre(c, Y, Z, sink);
    } else {  // with the centre last: 370 us a step of the Re 6500 nozzle instead of 354
        inverse_centre(c, Y, Z, sink);
        inverse_pair<1, 7>(c, Y, Z, sink);
        inverse_pair<3, 5>(c, Y, Z, sink);
        inverse_pair<0, 2>(c, Y, Z, sink);
        inverse_pair<6, 8>(c, Y, Z, sink);
    }
}

// The same moment sums axis by axis (x within a line, then y, then z), each
// +-1 pair summed and differenced once: 67 operations.  The form of FP64, the
// general collision and the FP32 / FP64 inlet/outlet nodes.
template <class R, class Load>
__device__ __forceinline__ void axis_sums(const Load &ld, R (&m)[10]) {
    R t0[3], e0[3], d0[3], t1[3], d1[3], t2[3];  // per cz: sums over cy of s0, s2-in-y, s1-in-y, ...
#pragma unroll
    for (int z = 0; z < 3; ++z) {
        R s0[3], s1[3], s2[3];
#pragma unroll
        for (int y = 0; y < 3; ++y) {
            const int j = 3 * (3 * z + y);
            const R a = ld(j), b = ld(j + 1), c = ld(j + 2);
            s2[y] = add_(c, a);
            s0[y] = add_(s2[y], b);
            s1[y] = sub_(c, a);
        }
        e0[z] = add_(s0[2], s0[0]);
        t0[z] = add_(e0[z], s0[1]);
        d0[z] = sub_(s0[2], s0[0]);
        t1[z] = add_(add_(s1[2], s1[0]), s1[1]);
        d1[z] = sub_(s1[2], s1[0]);
        t2[z] = add_(add_(s2[2], s2[0]), s2[1]);
    }
    m[6] = add_(t0[2], t0[0]);                  // pzz
    m[0] = add_(m[6], t0[1]);                   // drho
    m[1] = add_(add_(t1[2], t1[0]), t1[1]);     // jx
    m[2] = add_(add_(d0[2], d0[0]), d0[1]);     // jy
    m[3] = sub_(t0[2], t0[0]);                  // jz
    m[4] = add_(add_(t2[2], t2[0]), t2[1]);     // pxx
    m[5] = add_(add_(e0[2], e0[0]), e0[1]);     // pyy
    m[7] = add_(add_(d1[2], d1[0]), d1[1]);     // pxy
    m[8] = sub_(t1[2], t1[0]);                  // pxz
    m[9] = sub_(d0[2], d0[0]);                  // pyz
}

// The lines of ro f^eq/rho + sum k a_ab g_ab at velocity u, less the weights'
// part (ro - dro) w.  With ro = dro = 0 it gives the part of the relaxed
// second-order moments alone.  With the half coefficients
//   P0 = rho gz0 + Azz g2z, P1 = Ayz gz1, P2 = Ayy gz0   (cz level)
//   T = uy^2/2 P0 + uy P1 + P2/2,  O = (uy P0 + P1) / 2  (cy = +-1: +-O)
// a line's coefficients are Bd = gy0 P0 + gy1 P1 + g2y P2 = w P0 + T +- O and
// Bw = Bd - wy wz in the form w W0 + T +- O, W0 = rho dz + drho wz + Azz g2z,
// which has no O(1) cancellation; cy = 0 takes -2 T.  Along x, with
// u = ux^2/2 Bd + ux B1 + B2/2: f*_0 = 2/3 Bw - 2 u and f*_+- = Bw/6 + u
// +- (ux Bd + B1)/2.
template <class R, class Out>
__device__ __forceinline__ void relaxed_lines(R k, const R (&a2)[6], R ro, R dro, R ux, R uy, R uz, const Out &sink) {
    const R h = R(0.5), w0 = cst<R>(2, 3), w1_ = cst<R>(1, 6), m2 = R(-2), hk = mul_(h, k);
    const R hAxx = mul_(hk, a2[0]), hAyy = mul_(hk, a2[1]), hAzz = mul_(hk, a2[2]), nAzz = mul_(m2, hAzz);
    const R hAxy = mul_(hk, a2[3]), hAxz = mul_(hk, a2[4]), hAyz = mul_(hk, a2[5]);
    const R hux = mul_(h, ux), huy = mul_(h, uy), huz = mul_(h, uz);
    const R ux2h = mul_(hux, ux), uy2h = mul_(huy, uy), uz2h = mul_(huz, uz);
    const R u2x = mul_(R(2), ux), u2y = mul_(R(2), uy);
    const R gy0[3] = {add_(w1_, sub_(uy2h, huy)), fma_(m2, uy2h, w0), add_(w1_, add_(uy2h, huy))};
    const R gy1[3] = {sub_(uy, h), mul_(m2, uy), add_(uy, h)};
    const R Y1 = fma_(dro, w1_, hAzz), Y0 = fma_(dro, w0, nAzz);
#pragma unroll
    for (int z = 0; z < 3; ++z) {
        const R dz = z == 0 ? sub_(uz2h, huz) : (z == 1 ? mul_(m2, uz2h) : add_(uz2h, huz));
        const R gz0 = add_(z == 1 ? w0 : w1_, dz);
        const R gz1 = z == 0 ? sub_(uz, h) : (z == 1 ? mul_(m2, uz) : add_(uz, h));
        const R P0 = fma_(ro, gz0, z == 1 ? nAzz : hAzz), W0 = fma_(ro, dz, z == 1 ? Y0 : Y1);
        const R hP1 = mul_(hAyz, gz1), hP2 = mul_(hAyy, gz0);
        const R hQ0 = mul_(hAxz, gz1), hQ1 = mul_(hAxy, gz0), hR0 = mul_(hAxx, gz0);
        const R T = fma_(uy2h, P0, fma_(u2y, hP1, hP2)), O = fma_(huy, P0, hP1), n2T = mul_(m2, T);
        const R e1 = fma_(w1_, W0, T), e2 = fma_(w1_, P0, T);
#pragma unroll
        for (int y = 0; y < 3; ++y) {
            const R Bw = y == 0 ? sub_(e1, O) : (y == 1 ? fma_(w0, W0, n2T) : add_(e1, O));
            const R Bd = y == 0 ? sub_(e2, O) : (y == 1 ? fma_(w0, P0, n2T) : add_(e2, O));
            const R hB1 = fma_(gy0[y], hQ0, mul_(gy1[y], hQ1)), hB2 = mul_(gy0[y], hR0);
            const R u = fma_(ux2h, Bd, fma_(u2x, hB1, hB2));
            const R A = fma_(hux, Bd, hB1), S = fma_(w1_, Bw, u);
            sink(3 * z + y, sub_(S, A), fma_(m2, u, mul_(w0, Bw)), add_(S, A));
        }
    }
}

// The FP64 form of the second part.  FP64 is bound by its arithmetic pipe, so
// this form is the one with the fewest operations: the post-collision state
// is written in raw moments M_abc = sum c_x^a c_y^b c_z^c (f* - w) / 2^n, n
// the number of non-zero exponents, whose inverse is three operations a line
// (f*_+- = M_2 +- M_1, f*_0 = M_0 - 2 M_2) and holds no velocity.  With the
// 1-D moments (1, u, u^2 + theta) of the equilibrium factor and (0, 1, 2 u)
// of a first-order column, the 27 moments follow from rho, u and the relaxed
// second-order central moments A_ab = (1 - omega) a_ab, each from the ones
// of lower order:
//   p*_ab = p_ab - omega a_ab;  M(xxy) = u_y P_xx + 2 u_x A_xy, P = p* + theta;
//   M(xyz) = u_z p*_xy + u_y A_xz + u_x A_yz;
//   M(xxyy) = p*_xx E_y + A_yy E_x + 4 u_x u_y A_xy + theta u_y^2, E = u^2 + theta;
//   M(xxyz) = u_z M(xxy) + 2 u_x u_y A_xz + A_yz E_x;
//   M(xxyyz) = u_z (M(xxyy) + theta^2) + 2 u_x A_xz E_y + 2 u_y A_yz E_x; ...
// About 260 FP64 instructions a cell with the moment sums and the division,
// against about 390 for the line-by-line inverse; at the pipe's 86-87 % either
// way, the Re 3500 nozzle's step takes 2.12 ms instead of 3.12 ms (1 372 ->
// 2 030 MLUPS).
template <class R, class Out>
__device__ __forceinline__ void raw_finish(const R (&m)[10], R omega, R &rho, R &ux, R &uy, R &uz, const Out &sink) {
    const R drho = m[0], jx = m[1], jy = m[2], jz = m[3], th = theta0<R>(), h = R(0.5), q = R(0.25), m2 = R(-2);
    rho = add_(R(1), drho);
    const R inv = recip(rho);
    ux = mul_(jx, inv);
    uy = mul_(jy, inv);
    uz = mul_(jz, inv);
    const R a2[6] = {fma_(-jx, ux, fma_(-th, drho, m[4])), fma_(-jy, uy, fma_(-th, drho, m[5])),
                     fma_(-jz, uz, fma_(-th, drho, m[6])), fma_(-jx, uy, m[7]),
                     fma_(-jx, uz, m[8]),                  fma_(-jy, uz, m[9])};
    sink.moments(omega, a2);
    const R k = sub_(R(1), omega), hk = mul_(h, k);
    const R Axy = mul_(k, a2[3]), Axz = mul_(k, a2[4]), Ayz = mul_(k, a2[5]);
    const R hAyy = mul_(hk, a2[1]), hAzz = mul_(hk, a2[2]);
    const R qAxy = mul_(q, Axy), qAxz = mul_(q, Axz), qAyz = mul_(q, Ayz);
    const R hx = mul_(h, ux), hy = mul_(h, uy), hz = mul_(h, uz), u2y = add_(uy, uy), u2z = add_(uz, uz);
    const R sx = mul_(ux, ux), sy = mul_(uy, uy), sz = mul_(uz, uz);
    const R Ex = fma_(h, sx, R(h * th)), Ey = fma_(h, sy, R(h * th)), Ez = fma_(h, sz, R(h * th));
    const R ty = mul_(R(q * th), sy), tz = mul_(R(q * th), sz), t2 = R(q * th * th);
    const R kx_y = mul_(hx, Axy), ky_x = mul_(hy, Axy), kx_z = mul_(hx, Axz), kz_x = mul_(hz, Axz),
            ky_z = mul_(hy, Ayz), kz_y = mul_(hz, Ayz);
    R M[3][3][3];  // [a][b][c]
    M[0][0][0] = drho;
    M[1][0][0] = mul_(h, jx);
    M[0][1][0] = mul_(h, jy);
    M[0][0][1] = mul_(h, jz);
    M[2][0][0] = mul_(h, fma_(-omega, a2[0], m[4]));
    M[0][2][0] = mul_(h, fma_(-omega, a2[1], m[5]));
    M[0][0][2] = mul_(h, fma_(-omega, a2[2], m[6]));
    M[1][1][0] = mul_(q, fma_(-omega, a2[3], m[7]));
    M[1][0][1] = mul_(q, fma_(-omega, a2[4], m[8]));
    M[0][1][1] = mul_(q, fma_(-omega, a2[5], m[9]));
    const R Qxx = add_(M[2][0][0], R(h * th)), Qyy = add_(M[0][2][0], R(h * th)), Qzz = add_(M[0][0][2], R(h * th));
    M[2][1][0] = fma_(hy, Qxx, kx_y);
    M[2][0][1] = fma_(hz, Qxx, kx_z);
    M[1][2][0] = fma_(hx, Qyy, ky_x);
    M[0][2][1] = fma_(hz, Qyy, ky_z);
    M[1][0][2] = fma_(hx, Qzz, kz_x);
    M[0][1][2] = fma_(hy, Qzz, kz_y);
    M[1][1][1] = fma_(hz, M[1][1][0], fma_(hy, qAxz, mul_(hx, qAyz)));
    M[2][2][0] = fma_(M[2][0][0], Ey, fma_(hAyy, Ex, fma_(u2y, kx_y, ty)));
    M[2][0][2] = fma_(M[2][0][0], Ez, fma_(hAzz, Ex, fma_(u2z, kx_z, tz)));
    M[0][2][2] = fma_(M[0][2][0], Ez, fma_(hAzz, Ey, fma_(u2z, ky_z, tz)));
    M[2][1][1] = fma_(hz, M[2][1][0], fma_(hy, kx_z, mul_(qAyz, Ex)));
    M[1][2][1] = fma_(hz, M[1][2][0], fma_(hx, ky_z, mul_(qAxz, Ey)));
    M[1][1][2] = fma_(hy, M[1][0][2], fma_(hx, kz_y, mul_(qAxy, Ez)));
    const R T = fma_(kx_z, Ey, mul_(ky_z, Ex));
    M[2][2][1] = fma_(hz, add_(M[2][2][0], t2), T);
    M[2][1][2] = fma_(hy, add_(M[2][0][2], t2), fma_(kx_y, Ez, mul_(kz_y, Ex)));
    M[1][2][2] = fma_(hx, add_(M[0][2][2], t2), fma_(ky_x, Ez, mul_(kz_x, Ey)));
    M[2][2][2] = fma_(M[2][2][0], Ez, fma_(u2z, T, fma_(hAzz, mul_(Ex, Ey), mul_(R(h * th), tz))));
    // the inverse, axis by axis: index 0, 1, 2 is c = -1, 0, 1 afterwards
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const R n0 = M[a][b][0], n1 = M[a][b][1], n2 = M[a][b][2];
            M[a][b][0] = sub_(n2, n1);
            M[a][b][1] = fma_(m2, n2, n0);
            M[a][b][2] = add_(n2, n1);
        }
#pragma unroll
    for (int z = 0; z < 3; ++z) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const R n0 = M[a][0][z], n1 = M[a][1][z], n2 = M[a][2][z];
            M[a][0][z] = sub_(n2, n1);
            M[a][1][z] = fma_(m2, n2, n0);
            M[a][2][z] = add_(n2, n1);
        }
#pragma unroll
        for (int y = 0; y < 3; ++y) {
            const R n0 = M[0][y][z], n1 = M[1][y][z], n2 = M[2][y][z];
            sink(3 * z + y, sub_(n2, n1), fma_(m2, n2, n0), add_(n2, n1));
        }
    }
}

// Collision with the default ghost rates (all 1).  d holds f_i - w_i on entry;
// the post-collision f*_i - w_i go to the sink line by line.  rho, u receive
// the (conserved) moments.  With SCALED, d holds (f_i - w_i) / in_scale and the
// outputs are (f*_i - w_i) * out_scale.
template <class R, bool SCALED = false, class Out>
__device__ __forceinline__ void collide_ghost1(R (&d)[27], R omega, R &rho, R &ux, R &uy, R &uz, R in_scale, R out_scale,
                                               const Out &sink, Rounds rounds = Rounds()) {
    R m[10];
    auto ld = [&](int i) { return d[i]; };
    if constexpr (std::is_same<R, double>::value) {
        axis_sums<R>(ld, m);
        raw_finish<R>(m, omega, rho, ux, uy, uz, sink);
    } else {
        ghost1_sums<R>(ld, m);
        ghost1_finish<SCALED, R>(m, omega, rho, ux, uy, uz, in_scale, out_scale, SCALED ? rounds : Rounds(), sink);
    }
}

// The equilibrium part alone: the lines of ro f^eq(u)/rho less (ro - dro) w,
// plane by plane.  The weights of the x and y passes add up to 1 exactly, wq =
// (1 - w0) / 2: the FP32 roundings of 2/3 and 1/6 sum to 1 + 3e-8, each pass
// over them scales the momentum by that, and lattice BGK relaxes towards the
// result omega times a step.  (After 200 steps of the 64^3 vortex at Re 1600
// the velocity is off by 2.5e-5 with the rounded weights in every pass, by
// 1.3e-5, as with the cascade, with them in the z pass alone.)
template <class R>
struct EqLines {
    R ro, dro, hx, hy, hz, x2, y2, z2, Bw[3], Bd[3];
    __device__ __forceinline__ EqLines(R ro_, R dro_, R ux, R uy, R uz) : ro(ro_), dro(dro_) {
        const R h = R(0.5);
        hx = mul_(h, ux), hy = mul_(h, uy), hz = mul_(h, uz);
        x2 = mul_(hx, ux), y2 = mul_(hy, uy), z2 = mul_(hz, uz);
    }
    __device__ __forceinline__ void plane(int z) {  // cz = z - 1
        const R w0 = cst<R>(2, 3), wp = cst<R>(1, 6), wq = (R(1) - w0) / R(2), m2 = R(-2), wz = z == 1 ? w0 : wp;
        const R dz = z == 0 ? sub_(z2, hz) : (z == 1 ? mul_(m2, z2) : add_(z2, hz));
        const R P0 = mul_(ro, add_(wz, dz)), W0 = fma_(ro, dz, mul_(dro, wz));
        const R T = mul_(y2, P0), O = mul_(hy, P0), n2T = mul_(m2, T), e1 = fma_(wq, W0, T), e2 = fma_(wq, P0, T);
        Bw[0] = sub_(e1, O), Bw[1] = fma_(w0, W0, n2T), Bw[2] = add_(e1, O);
        Bd[0] = sub_(e2, O), Bd[1] = fma_(w0, P0, n2T), Bd[2] = add_(e2, O);
    }
    __device__ __forceinline__ void line(int y, R &vm, R &v0, R &vp) const {  // cy = y - 1 of the current plane
        const R w0 = cst<R>(2, 3), wq = (R(1) - w0) / R(2);
        const R t = mul_(x2, Bd[y]), S = fma_(wq, Bw[y], t), A = mul_(hx, Bd[y]);
        vm = sub_(S, A);
        v0 = fma_(R(-2), t, mul_(w0, Bw[y]));
        vp = add_(S, A);
    }
};

// Collision with every ghost rate equal to omega.  T^-1 S T is then omega on
// all but the conserved moments, on which f^eq - f has no part, so the step
// is lattice BGK with the full equilibrium (Sec. 2.1): f* = f + omega (f^eq
// - f), in deviations, with the equilibrium's lines as in relaxed_lines.
// About 250 operations instead of 600 for the 27-moment cascade, and no 27
// moments to hold.
template <class R, class Out>
__device__ __forceinline__ void collide_bgk(R (&d)[27], R omega, R &rho, R &ux, R &uy, R &uz, const Out &sink) {
    R m[10];
    ghost1_sums<R>([&](int i) { return d[i]; }, m);
    const R drho = m[0], jx = m[1], jy = m[2], jz = m[3], th = theta0<R>();
    rho = add_(R(1), drho);
    const R inv = recip(rho);
    ux = mul_(jx, inv);
    uy = mul_(jy, inv);
    uz = mul_(jz, inv);
    const R a2[6] = {fma_(-jx, ux, fma_(-th, drho, m[4])), fma_(-jy, uy, fma_(-th, drho, m[5])),
                     fma_(-jz, uz, fma_(-th, drho, m[6])), fma_(-jx, uy, m[7]),
                     fma_(-jx, uz, m[8]),                  fma_(-jy, uz, m[9])};
    sink.moments(omega, a2);  // unused but for statistics
    const R keep = sub_(R(1), omega);
    EqLines<R> eq(mul_(rho, omega), mul_(drho, omega), ux, uy, uz);  // omega on the equilibrium's two coefficients
#pragma unroll
    for (int z = 0; z < 3; ++z) {
        eq.plane(z);
#pragma unroll
        for (int y = 0; y < 3; ++y) {
            const int j = 3 * z + y;
            R vm, v0, vp;
            eq.line(y, vm, v0, vp);
            sink(j, fma_(keep, d[3 * j], vm), fma_(keep, d[3 * j + 1], v0), fma_(keep, d[3 * j + 2], vp));
        }
    }
}

// One axis of T(u) on a line of three values: the sums weighted by 1, c - u
// and (c - u)^2 - theta0.  And back.
template <class R>
__device__ __forceinline__ void to_central(R u, R &lo, R &mid, R &hi) {
    const R s = add_(hi, lo), d = sub_(hi, lo);
    const R m0 = add_(s, mid), m1 = fma_(-u, m0, d);
    hi = fma_(-theta0<R>(), m0, fma_(-u, add_(d, m1), s));
    mid = m1;
    lo = m0;
}
template <class R>
__device__ __forceinline__ void from_central(R u, R &a0, R &a1, R &a2) {
    const R n1 = fma_(u, a0, a1);               // first raw moment
    const R x = fma_(u, add_(a1, n1), a2);      // second one less theta0 a0
    const R t = fma_(cst<R>(1, 6), a0, mul_(R(0.5), x));
    a1 = fma_(cst<R>(2, 3), a0, -x);
    a0 = fma_(R(-0.5), n1, t);
    a2 = fma_(R(0.5), n1, t);
}

// Collision with general ghost rates: the full 27-moment cascade, in place.
//   dA = T(u) (f - w), A = e(u) + dA with e_m = prod_a e_{m_a}(u_a),
//   e0 = 1, e1 = -u, e2 = u^2 (the central moments of the weights);
//   A* = A + S (A^eq - A), A^eq = (rho, 0, ..., 0);
//   f* - w = T^-1 (A* - e), A* - e = (1 - s) dA - s e for orders 2 and more.
template <class R, class Sink = ToArray<R>>
__device__ __forceinline__ void collide_general(R (&d)[27], R omega, const R (&ghost)[4], R &rho, R &ux,
                                                R &uy, R &uz, const Sink *sink = nullptr) {
    R s[10];
    axis_sums<R>([&](int i) { return d[i]; }, s);
    const R drho = s[0];
    rho = add_(R(1), drho);
    const R inv = recip(rho);
    ux = mul_(s[1], inv);
    uy = mul_(s[2], inv);
    uz = mul_(s[3], inv);
#pragma unroll
    for (int j = 0; j < 9; ++j) to_central(ux, d[3 * j], d[3 * j + 1], d[3 * j + 2]);
#pragma unroll
    for (int k = 0; k < 9; ++k) {  // (kx, cz)
        const int b = k % 3 + 9 * (k / 3);
        to_central(uy, d[b], d[b + 3], d[b + 6]);
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) to_central(uz, d[k], d[k + 9], d[k + 18]);
    if (sink) {  // second-order central Hermite moments A_m = e_m + dA_m
        const R a2[6] = {fma_(ux, ux, d[2]), fma_(uy, uy, d[6]),  fma_(uz, uz, d[18]),
                         fma_(ux, uy, d[4]), fma_(ux, uz, d[10]), fma_(uy, uz, d[12])};
        sink->moments(omega, a2);
    }
    const R ex[3] = {R(1), -ux, mul_(ux, ux)}, ey[3] = {R(1), -uy, mul_(uy, uy)}, ez[3] = {R(1), -uz, mul_(uz, uz)};
#pragma unroll
    for (int m = 0; m < 27; ++m) {
        const int kx = m % 3, ky = (m / 3) % 3, kz = m / 9, n = kx + ky + kz;
        const R exy = kx == 0 ? ey[ky] : (ky == 0 ? ex[kx] : mul_(ex[kx], ey[ky]));
        const R e = kz == 0 ? exy : (kx + ky == 0 ? ez[kz] : mul_(exy, ez[kz]));
        if (n == 0) {
            d[m] = drho;  // A*_0 = rho, e_0 = 1
        } else if (n == 1) {
            d[m] = -e;    // A*_1 = 0
        } else {
            const R rate = n == 2 ? omega : ghost[n - 3];
            d[m] = fma_(sub_(R(1), rate), d[m], -mul_(rate, e));
        }
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) from_central(uz, d[k], d[k + 9], d[k + 18]);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const int b = k % 3 + 9 * (k / 3);
        from_central(uy, d[b], d[b + 3], d[b + 6]);
    }
#pragma unroll
    for (int j = 0; j < 9; ++j) from_central(ux, d[3 * j], d[3 * j + 1], d[3 * j + 2]);
}

// ---------------------------------------------------------------- streaming

// The nine neighbour-row bases of a row record (j = (cy+1) + 3 (cz+1)).
__device__ __forceinline__ void load_row(const int4 *row_nb, int row, int (&nb)[9]) {
    const int4 a = __ldg(row_nb + 3 * row), b = __ldg(row_nb + 3 * row + 1), c = __ldg(row_nb + 3 * row + 2);
    nb[0] = a.x; nb[1] = a.y; nb[2] = a.z; nb[3] = a.w;
    nb[4] = b.x; nb[5] = b.y; nb[6] = b.z; nb[7] = b.w;
    nb[8] = c.x;
}

// Element offset of (population i, slot s): i * stride + s, in 32-bit
// unsigned arithmetic when the buffer allows (see MAX_SLOTS_32).
template <bool WIDE>
__device__ __forceinline__ typename std::conditional<WIDE, int64_t, uint32_t>::type
elem(int i, int64_t stride, int s) {
    if constexpr (WIDE)
        return (int64_t)i * stride + s;
    else
        return (uint32_t)i * (uint32_t)stride + (uint32_t)s;
}

// Pull gather of the cell at x in the row with bases nb: d_i = f*_i(x - c_i)
// from slot nb[j] + x - cx of population array i.  For a wall link that slot
// is the ghost slot holding f*_{26-i}(x) (halfway bounce-back, i.e.
// Bouzidi's interpolated bounce-back at q = 1/2, Sec. 2.2).
template <int P, bool WIDE, int AX, bool RAW = false, bool CG = false>
__device__ __forceinline__ void gather(const StepArgs &a, const int (&nb)[9], int x, typename Storage<P>::R (&d)[27]) {
    using S = Storage<P>;
    using T = typename S::T;
    using R = typename S::R;
    const T *fin = static_cast<const T *>(a.fin);
    const R inv_s = R(a.inv_scale);
#if LBM_LINE_POINTERS
    if constexpr (!WIDE && P == 2) {
        // one pointer per storage line j (its three populations pull from
        // row nb[j]); the pulls sit at +1, +(k1 - k0) stride, +(k2 - k0) stride - 1
        const uint32_t st = (uint32_t)a.stride;
#pragma unroll
        for (int j = 0; j < 9; ++j) {
            constexpr int dk = line_pop<AX>(0, 1) - line_pop<AX>(0, 0);
            const T *pj = fin + ((uint32_t)line_pop<AX>(j, 0) * st + (uint32_t)(nb[j] + x));
            const T *q[3] = {pj + 1, pj + dk * st, pj + 2 * dk * st - 1};
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int i = line_pop<AX>(j, k);
                d[i] = RAW ? S::template load_raw<CG>(q[k]) : S::template load<CG>(q[k], inv_s);
            }
        }
        return;
    }
#endif
#pragma unroll
    for (int i = 0; i < 27; ++i) {
        const T *p = fin + elem<WIDE>(i, a.stride, nb[row_line<AX>(i)] + x - c_row<AX>(i));
        d[i] = RAW ? S::template load_raw<CG>(p) : S::template load<CG>(p, inv_s);  // RAW: storage value, scale applied later
    }
}

// Bouzidi's interpolated bounce-back (Sec. 2.2) on the wall links of a cell
// whose wall distances were given (lbm_set_wall_q).  The gather has already
// put f*_ib(x) into d[i] for every wall link i (the ghost slot, halfway
// bounce-back; ib = 26 - i is the direction from x towards the wall), and the
// pull of ib into d[ib].  With q the wall's distance from x as a fraction of
// the link:
//   q <  1/2: f_i = 2q f*_ib(x) + (1 - 2q) f*_ib(x + c_i)   (= d[ib], unless
//             x + c_i is a wall too: then the halfway value stays),
//   q >= 1/2: f_i = f*_ib(x) / (2q) + (1 - 1/(2q)) f*_i(x)   (own slot, array i).
// Every term is a deviation (or scaled deviation) from w_i = w_ib, and the
// coefficients sum to 1, so the storage form needs no conversion.
template <int P, bool WIDE, bool RAW, bool CG = false>
__device__ __forceinline__ void interpolate_walls(const StepArgs &a, int k, int slot, uint32_t links,
                                                  typename Storage<P>::R (&d)[27]) {
    using S = Storage<P>;
    using T = typename S::T;
    using R = typename S::R;
    if (k < 0) return;
    // the record as two 16-byte loads; byte i = q of link i in 1/256
    const uint4 *rec = reinterpret_cast<const uint4 *>(a.wall_q) + 2 * (size_t)k;
    const uint4 r0 = __ldg(rec), r1 = __ldg(rec + 1);
    const uint32_t w[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
    const T *fin = static_cast<const T *>(a.fin);
    // own-slot values for the links with q > 1/2, all loads issued first
    R own[27];
#pragma unroll
    for (int i = 0; i < 27; ++i) {
        const uint32_t q8 = (w[i >> 2] >> (8 * (i & 3))) & 0xFFu;
        own[i] = R(0);
        if ((links & (1u << i)) && q8 > 128u) {
            const T *p = fin + elem<WIDE>(i, a.stride, slot);
            own[i] = RAW ? S::template load_raw<CG>(p) : S::template load<CG>(p, R(a.inv_scale));
        }
    }
#pragma unroll
    for (int i = 0; i < 27; ++i) {
        if (!(links & (1u << i))) continue;
        const uint32_t q8 = (w[i >> 2] >> (8 * (i & 3))) & 0xFFu;
        const int ib = 26 - i;
        if (q8 < 128u) {
            if (links & (1u << ib)) continue;
            const R q2 = R(q8) * R(1.0 / 128.0);  // 2q
            d[i] = fma_(q2, d[i], mul_(sub_(R(1), q2), d[ib]));
        } else if (q8 > 128u) {
            const R c = R(128) / R(q8);  // 1 / (2q)
            d[i] = fma_(c, d[i], mul_(sub_(R(1), c), own[i]));
        }
    }
}

// ------------------------------------------------------------------- inlet

__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
    // SplitMix64 output function (Steele, Lea and Flood 2014).
    uint64_t z = x + 0x9e3779b97f4a7c15ULL;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
    return z ^ (z >> 31);
}

// Counter-based uniform variate in [-1, 1) for (seed, step, node, component);
// 24 random bits, exact in binary32.
template <class R>
__device__ __forceinline__ R inlet_noise(uint64_t seed, int64_t step, int64_t node, int comp) {
    uint64_t h = splitmix64(seed);
    h = splitmix64((uint64_t)step + h);
    h = splitmix64((((uint64_t)node << 2) | (uint64_t)comp) + h);
    return fma_(R((uint32_t)(h >> 40)), R(1.0 / 8388608.0), R(-1));
}

// -------------------------------------------------------- block reduction

__device__ __forceinline__ void block_reduce_write(double (&v)[6], double *partials) {
    __shared__ double sh[32][6];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const double t = __shfl_down_sync(0xffffffffu, v[k], o);
            v[k] = (k == 4) ? fmax(v[k], t) : v[k] + t;
        }
    }
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < 6; ++k) sh[warp][k] = v[k];
    __syncthreads();
    if (threadIdx.x == 0) {
        double r[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) r[k] = sh[0][k];
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w)
#pragma unroll
            for (int k = 0; k < 6; ++k) r[k] = (k == 4) ? fmax(r[k], sh[w][k]) : r[k] + sh[w][k];
        double *p = partials + (size_t)blockIdx.x * REDUCE_SLOTS;
#pragma unroll
        for (int k = 0; k < 6; ++k) p[k] = r[k];
    }
}

__device__ __forceinline__ void health_values(double rho, double ux, double uy, double uz, double (&v)[6]) {
    const bool finite = isfinite(rho) && isfinite(ux) && isfinite(uy) && isfinite(uz);
    v[0] = rho;
    v[1] = rho * ux;
    v[2] = rho * uy;
    v[3] = rho * uz;
    v[4] = finite ? sqrt(ux * ux + uy * uy + uz * uz) : 0.0;
    v[5] = finite ? 0.0 : 1.0;
}

// --------------------------------------------------------------- step kernel

template <class R>
__device__ __forceinline__ const FlowParams<R> &flow(const StepArgs &a);
template <>
__device__ __forceinline__ const FlowParams<double> &flow<double>(const StepArgs &a) { return a.pd; }
template <>
__device__ __forceinline__ const FlowParams<float> &flow<float>(const StepArgs &a) { return a.pf; }

// Collision of d in place; the viscous stress is recorded at stress_slot.
template <int P, int G>
__device__ __forceinline__ void collide(typename Storage<P>::R (&d)[27], const FlowParams<typename Storage<P>::R> &fp,
                                        typename Storage<P>::R &rho, typename Storage<P>::R &ux,
                                        typename Storage<P>::R &uy, typename Storage<P>::R &uz, const StepArgs &a,
                                        int stress_slot) {
    using R = typename Storage<P>::R;
    const ToArrayStress<R> sink{a, stress_slot, d};
    if constexpr (G == RATE_ONE)
        collide_ghost1<R>(d, fp.omega, rho, ux, uy, uz, R(1), R(1), sink);
    else if constexpr (G == RATE_BGK)
        collide_bgk<R>(d, fp.omega, rho, ux, uy, uz, sink);
    else
        collide_general<R, ToArrayStress<R>>(d, fp.omega, fp.ghost, rho, ux, uy, uz, &sink);
}

// Post-collision state of one cell is in d; write it to its own slot, the
// ghost slots of its wall links, and (periodic row axis) its wrap-around
// copies.
template <int P, bool WIDE, int AX, bool RAW = false>
__device__ __forceinline__ void store_cell_state(const StepArgs &a, const int (&nb)[9], int x, int slot, uint32_t links,
                                                 const typename Storage<P>::R (&d)[27]) {
    using S0 = Storage<P>;
    using T = typename S0::T;
    using R = typename S0::R;
    // RAW: d already holds storage values (scale applied by the collision)
    struct S {
        static __device__ __forceinline__ void store(T *p, R v, R sc) {
            if constexpr (RAW)
                S0::store_raw(p, v);
            else
                S0::store(p, v, sc);
        }
    };
    const R s = R(a.scale);
    T *fout = static_cast<T *>(a.fout);
#pragma unroll
    for (int i = 0; i < 27; ++i) S::store(fout + elem<WIDE>(i, a.stride, slot), d[i], s);
    if (links) {  // wall links: the reflected population waits in the ghost slot
#pragma unroll
        for (int j = 0; j < 9; ++j) {
            if (!(links & (7u << (3 * j)))) continue;  // no wall link among populations 3j .. 3j + 2
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int i = 3 * j + c;
                if (links & (1u << i))
                    S::store(fout + elem<WIDE>(i, a.stride, nb[row_line<AX>(i)] + x - c_row<AX>(i)), d[26 - i], s);
            }
        }
    }
    if (a.periodic_row) {  // wrap-around copies read across the periodic faces of the row axis
        if (x == a.n_row - 1) {
#pragma unroll
            for (int i = 0; i < 27; ++i)
                if (c_row<AX>(i) == 1) S::store(fout + elem<WIDE>(i, a.stride, nb[4] - 1), d[i], s);
        }
        if (x == 0) {
#pragma unroll
            for (int i = 0; i < 27; ++i)
                if (c_row<AX>(i) == -1) S::store(fout + elem<WIDE>(i, a.stride, nb[4] + a.n_row), d[i], s);
        }
    }
}

// Output sink of the fluid update: each line of three post-collision values
// (populations 3j .. 3j + 2) goes to the cell's own slots at once, to the
// ghost slots of the wall links they serve (value i feeds link 26 - i), and
// across a periodic face of the row axis.
// own: bit i set = store value i in the cell's own slot; bit 31 = the lane is
// a fluid cell (the other lanes only fill unread arrays, see fluid_cell).
constexpr uint32_t OWN_FLUID = 1u << 31;

template <int P, bool WIDE, bool RAW, int AX>
struct LineStore {
    using S = Storage<P>;
    using T = typename S::T;
    using R = typename S::R;
    const StepArgs &a;
    const int (&nb)[9];
    int x, slot;
    uint32_t links, own;
    __device__ __forceinline__ void put(int i, int s, R v) const {
        T *p = static_cast<T *>(a.fout) + elem<WIDE>(i, a.stride, s);
        if constexpr (RAW)
            S::store_raw(p, v);
        else
            S::store(p, v, R(a.scale));
    }
    __device__ __forceinline__ void moments(R omega, const R (&a2)[6]) const {
        if (own & OWN_FLUID) record_stress(a, slot, omega, a2);
    }
    __device__ __forceinline__ void operator()(int j, R vm, R v0, R vp) const {
#if LBM_LINE_POINTERS
        if constexpr (!WIDE && P == 2) {  // the three own-slot stores of line j from one pointer
            const uint32_t st = (uint32_t)a.stride;
            T *pj = static_cast<T *>(a.fout) + ((uint32_t)(3 * j) * st + (uint32_t)slot);
            const R v[3] = {vm, v0, vp};
            T *q[3] = {pj, pj + st, pj + 2 * st};
#pragma unroll
            for (int c = 0; c < 3; ++c)
                if (own & (1u << (3 * j + c))) {
                    if constexpr (RAW)
                        S::store_raw(q[c], v[c]);
                    else
                        S::store(q[c], v[c], R(a.scale));
                }
        } else
#endif
        {
            if (own & (1u << (3 * j))) put(3 * j, slot, vm);
            if (own & (2u << (3 * j))) put(3 * j + 1, slot, v0);
            if (own & (4u << (3 * j))) put(3 * j + 2, slot, vp);
        }
        const int jl = 8 - j;  // links 26 - i of this line's values sit in line 8 - j
        if (links & (7u << (3 * jl))) {
            const R v[3] = {vm, v0, vp};
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int k = 26 - (3 * j + c);  // wall link k takes value 3j + c
                if (links & (1u << k)) put(k, nb[row_line<AX>(k)] + x - c_row<AX>(k), v[c]);
            }
        }
        if (a.periodic_row && (own & OWN_FLUID)) {  // wrap-around copies across the periodic row faces
            const R v[3] = {vm, v0, vp};
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int i = 3 * j + c;
                if (c_row<AX>(i) == 1 && x == a.n_row - 1) put(i, nb[4] - 1, v[c]);
                if (c_row<AX>(i) == -1 && x == 0) put(i, nb[4] + a.n_row, v[c]);
            }
        }
    }
};

// Output sink of the fast path (a warp of fluid cells without wall links):
// the 27 post-collision values go to the cell's own slots only, with no
// predicate.  FP16S addresses each line's three stores from one pointer, FP32
// by per-population offsets, as LineStore does.
template <int P, bool RAW>
struct OwnStore {
    using S = Storage<P>;
    using T = typename S::T;
    using R = typename S::R;
    const StepArgs &a;
    int slot;
    __device__ __forceinline__ void put(T *p, R v) const {
        if constexpr (RAW)
            S::store_raw(p, v);
        else
            S::store(p, v, R(a.scale));
    }
    __device__ __forceinline__ void moments(R omega, const R (&a2)[6]) const { record_stress(a, slot, omega, a2); }
    __device__ __forceinline__ void operator()(int j, R vm, R v0, R vp) const {
        T *out = static_cast<T *>(a.fout);
        const uint32_t st = (uint32_t)a.stride;
        if constexpr (LBM_LINE_POINTERS && P == 2) {
            T *pj = out + ((uint32_t)(3 * j) * st + (uint32_t)slot);
            put(pj, vm);
            put(pj + st, v0);
            put(pj + 2 * st, vp);
        } else {
            put(out + elem<false>(3 * j, a.stride, slot), vm);
            put(out + elem<false>(3 * j + 1, a.stride, slot), v0);
            put(out + elem<false>(3 * j + 2, a.stride, slot), vp);
        }
    }
};

template <class R>
__device__ __forceinline__ void record_axial(const StepArgs &a, int slot, R uz) {
    const double w = (double)uz;
    a.stats[slot] += w;
    a.stats[a.stride + slot] = fma_(w, w, a.stats[a.stride + slot]);
}

template <class R>
__device__ __forceinline__ void record_cell(const StepArgs &a, int slot, R rho, R ux, R uy, R uz, double (&hv)[6]) {
    if (a.flags & STEP_STATS) {
        record_axial(a, slot, uz);
        if (a.flags & STEP_STATS_FULL) {  // time averages of u, u u and rho (Sec. 2.2)
            const double u[3] = {(double)ux, (double)uy, (double)uz};
            double *p = a.stats + 2 * (int64_t)a.stride + slot;
#pragma unroll
            for (int q = 0; q < 3; ++q) p[q * a.stride] += u[q];
#pragma unroll
            for (int q = 0; q < 6; ++q) {  // xx, yy, zz, xy, xz, yz
                const int x = q < 3 ? q : (q == 5 ? 1 : 0), y = q < 3 ? q : (q == 3 ? 1 : 2);
                p[(3 + q) * a.stride] = fma_(u[x], u[y], p[(3 + q) * a.stride]);
            }
            p[15 * a.stride] += (double)rho;
        }
    }
    if (a.flags & STEP_REDUCE) health_values(rho, ux, uy, uz, hv);
}

// Update of the fluid cell in lane `lane` of chunk `chunk` (Sec. 2.1
// evolution equation, pull form): gather, collide, store, refill the ghost
// slots of its wall links.  The chunk's other lanes run the same instruction
// stream on whatever their pull slots hold (all inside the buffer and its
// margins) and store the result only into the arrays that nobody reads at
// their slot (link word of a padding / ghost slot: bit i = array i is read
// there; nothing at inlet/outlet slots).  This completes the 32-byte sectors
// at the row ends, which the memory system would otherwise have to read
// back before writing them, at no extra instructions per warp.
template <int P, int G, bool WIDE, bool WALLQ, int AX, bool CG = false>
__device__ __forceinline__ void cell_update(const StepArgs &a, int row, int x, bool fluid, bool plain, int qk, double (&hv)[6]) {
    using R = typename Storage<P>::R;
    int nb[9];
    load_row(a.row_nb, row, nb);
    const int slot = nb[4] + x;
    const uint32_t m = __ldg(a.mask + slot);  // needed after the collision only
    const uint32_t links = fluid ? (m & LINK_MASK) : 0u;
    const uint32_t own = fluid ? (LINK_MASK | OWN_FLUID)
                               : (((m >> TYPE_SHIFT) & 3u) == TYPE_PAD ? (~m & LINK_MASK) : 0u);
    R d[27];
    R rho, ux, uy, uz;
    constexpr bool RAW = G == RATE_ONE && Storage<P>::SCALED;  // FP16 scale folded into the collision
    gather<P, WIDE, AX, RAW, CG>(a, nb, x, d);
    if constexpr (WALLQ) interpolate_walls<P, WIDE, RAW, CG>(a, qk, slot, links, d);
    if constexpr (G != RATE_GENERAL) {
        const LineStore<P, WIDE, RAW, AX> sink{a, nb, x, slot, links, own};
        if constexpr (G == RATE_ONE)
            collide_ghost1<R, RAW>(d, flow<R>(a).omega, rho, ux, uy, uz, R(a.inv_scale), R(a.scale), sink,
                                   lane_rounds<AX>(plain));
        else
            collide_bgk<R>(d, flow<R>(a).omega, rho, ux, uy, uz, sink);
    } else {
        if (!fluid) return;
        collide<P, G>(d, flow<R>(a), rho, ux, uy, uz, a, slot);
        store_cell_state<P, WIDE, AX, RAW>(a, nb, x, slot, links, d);
    }
    if (fluid) record_cell(a, slot, rho, ux, uy, uz, hv);
}

template <int P, int G, bool WIDE, int AX, bool CG = false>
__device__ __forceinline__ void fluid_cell(const StepArgs &a, int chunk, int lane, double (&hv)[6]) {
    const int2 ch = __ldg(a.chunks + chunk);
    const uint32_t cw = (uint32_t)ch.y;
    const bool fluid = (cw >> (CHUNK_LANES_SHIFT + lane)) & 1u;
    cell_update<P, G, WIDE, false, AX, CG>(a, ch.x, (int)(cw & CHUNK_X0_MASK) + lane, fluid, cw & CHUNK_PLAIN, -1, hv);
}

// Fluid lane of the step kernel with a warp-uniform fast path (default ghost
// rates, 32-bit offsets, FP32 / FP16S).  With rows along the flow axis most
// warps hold 32 fluid cells none of which has a wall link (or, on a periodic
// row axis, sits at a row end); such a warp stores every cell's 27 values
// into its own slots and skips the line sink's per-value predicates,
// ghost-slot stores and wrap-around copies.  The gather is the same on both paths, so it
// is issued before the vote.  Every lane of the warp must call this (lanes
// past the last chunk take part in the vote only).
template <int P, int G, int AX>
__device__ __forceinline__ void fluid_lane_voted(const StepArgs &a, int chunk, int lane, double (&hv)[6]) {
    using R = typename Storage<P>::R;
    constexpr bool RAW = Storage<P>::SCALED;
    const bool valid = chunk < a.nchunks;
    int nb[9];
    R d[27];
    int x = 0, slot = 0;
    uint32_t m = 0u;
    bool fluid = false, plain = false;
    if (valid) {
        const int2 ch = __ldg(a.chunks + chunk);
        const uint32_t cw = (uint32_t)ch.y;
        fluid = (cw >> (CHUNK_LANES_SHIFT + lane)) & 1u;
        plain = cw & CHUNK_PLAIN;
        x = (int)(cw & CHUNK_X0_MASK) + lane;
        load_row(a.row_nb, ch.x, nb);
        slot = nb[4] + x;
        gather<P, false, AX, RAW>(a, nb, x, d);
        m = __ldg(a.mask + slot);
    }
    const bool row_end = a.periodic_row && (x == 0 || x == a.n_row - 1);  // writes wrap-around copies
    const bool simple = fluid && (m & LINK_MASK) == 0u && !row_end;
    const bool fast = __all_sync(0xffffffffu, simple);
    if (!valid) return;
    R rho, ux, uy, uz;
    if (fast) {
        const OwnStore<P, RAW> sink{a, slot};
        collide_ghost1<R, RAW>(d, flow<R>(a).omega, rho, ux, uy, uz, R(a.inv_scale), R(a.scale), sink, lane_rounds<AX>(plain));
    } else {
        const uint32_t links = fluid ? (m & LINK_MASK) : 0u;
        const uint32_t own = fluid ? (LINK_MASK | OWN_FLUID)
                                   : (((m >> TYPE_SHIFT) & 3u) == TYPE_PAD ? (~m & LINK_MASK) : 0u);
        const LineStore<P, false, RAW, AX> sink{a, nb, x, slot, links, own};
        collide_ghost1<R, RAW>(d, flow<R>(a).omega, rho, ux, uy, uz, R(a.inv_scale), R(a.scale), sink, lane_rounds<AX>(plain));
    }
    if (fluid) record_cell(a, slot, rho, ux, uy, uz, hv);
}

// Update of wall cell k of the interpolated-wall list (x, row, slot, record):
// the same update with Bouzidi's interpolation of its wall links.  These
// cells are taken out of the chunk lanes while wall distances are set, so
// the fluid kernel keeps its plain instruction stream.
template <int P, int G, bool WIDE, int AX, bool CG = false>
__device__ __forceinline__ void wall_cell(const StepArgs &a, int k, double (&hv)[6]) {
    const int4 node = __ldg(a.wnodes + k);
    cell_update<P, G, WIDE, true, AX, CG>(a, node.y, node.x, true, true, node.w, hv);
}

// Output sink of an inlet/outlet node: f* - f^eq of the partner comes in, the
// node's own equilibrium is added, and the values go to its own slots and, at
// a row end of a periodic row axis, the wrap-around copies.
template <int P, bool WIDE, int AX>
struct NodeStore {
    using S = Storage<P>;
    using T = typename S::T;
    using R = typename S::R;
    const StepArgs &a;
    int slot, pos;
    mutable EqLines<R> eq;
    __device__ __forceinline__ void put(int i, int s, R v) const {
        S::store(static_cast<T *>(a.fout) + elem<WIDE>(i, a.stride, s), v, R(a.scale));
    }
    __device__ __forceinline__ void moments(R omega, const R (&a2)[6]) const {}
    __device__ __forceinline__ void operator()(int j, R vm, R v0, R vp) const {
        R e[3];
        if (j % 3 == 0) eq.plane(j / 3);
        eq.line(j % 3, e[0], e[1], e[2]);
        line(j, add_(vm, e[0]), add_(v0, e[1]), add_(vp, e[2]));
    }
    __device__ __forceinline__ void line(int j, R vm, R v0, R vp) const {
        const R v[3] = {vm, v0, vp};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const int i = 3 * j + c;
            put(i, slot, v[c]);
            if (a.periodic_row) {
                if (c_row<AX>(i) == 1 && pos == a.n_row - 1) put(i, slot - pos - 1, v[c]);
                if (c_row<AX>(i) == -1 && pos == 0) put(i, slot + a.n_row, v[c]);
            }
        }
    }
};

// One line (cx = -1, 0, 1) of f^eq(rho, u) - w in product form, without O(1)
// cancellation: (rho - 1) w + rho (dx gy gz + wx (dy gz + wy dz)).  The FP16S
// nodes' form, with one set of roundings as in Rounds.
struct EqNode {
    Axis<float> X, Y, Z;
    float r, dr;
    __device__ __forceinline__ EqNode(float rho, float ux, float uy, float uz)
        : X(ux, false, false), Y(uy, false, false), Z(uz, false, false), r(rho), dr(sub_(rho, 1.0f)) {}
    __device__ __forceinline__ void line(int j, float (&e)[3]) const {
        const int y = j % 3, z = j / 3;
        const float wy = w1<float>(y - 1), E = mul_(Y.g0[y], Z.g0[z]);
        const float D = y == 1 ? fma_(wy, Z.d[z], mul_(Y.d[y], Z.g0[z])) : fma_(Y.d[y], Z.g0[z], mul_(wy, Z.d[z]));
#pragma unroll
        for (int x = 0; x < 3; ++x) {
            const float wx = w1<float>(x - 1), ww = wx * wy * w1<float>(z - 1), p = fma_(wx, D, mul_(X.d[x], E));
            e[x] = j == 4 && x == 1 ? fma_(dr, ww, mul_(r, p)) : fma_(r, p, mul_(dr, ww));
        }
    }
};

// Update of inlet/outlet node k: non-equilibrium extrapolation (Sec. 2.2)
// from the interior partner x_f, whose update is recomputed here from the
// same input state (so boundary and fluid updates are independent):
//   f*_i(x_b) = f^eq_i(rho_b, u_b) + f*_i(x_f) - f^eq_i(rho_f, u_f),
// inlet: rho_b = rho_f, u_b prescribed; outlet: rho_b = rho_out, u_b = u_f.
// With the default rates f* - f^eq of the partner is its relaxed
// second-order part alone, so no equilibrium of the partner is formed (FP16S
// forms both, see Rounds).
// Few nodes run at a time, each a chain of latencies; what counts is the
// depth of the dependent loads (record, pulls) and the operations after
// them.
template <int P, int G, bool WIDE, int AX, bool CG = false>
__device__ __forceinline__ void boundary_node(const StepArgs &a, int k, double (&hv)[6]) {
    using R = typename Storage<P>::R;
    const int4 *rec = a.bnodes + (size_t)NODE_INT4S * k;
    const int4 r0 = __ldg(rec), r1 = __ldg(rec + 1), r2 = __ldg(rec + 2), r3 = __ldg(rec + 3), r4 = __ldg(rec + 4);
    const int slot = r0.x, pos = r0.z, pf = r0.w;
    const uint32_t m = (uint32_t)r0.y;
    const int nbf[9] = {r2.x, r2.y, r2.z, r2.w, r3.x, r3.y, r3.z, r3.w, r4.x};
    const FlowParams<R> &fp = flow<R>(a);
    R d[27];
    gather<P, WIDE, AX, false, CG>(a, nbf, pf, d);
    const bool inlet = ((m >> TYPE_SHIFT) & 3u) == TYPE_INLET;
    R ux = R(0), uy = R(0), uz = R(0);  // the inlet's prescribed velocity, while the pulls are under way
    if (inlet) {
        const int dir = (int)(m >> DIR_SHIFT);
        R speed = fp.u_in;
        if (a.profile == LBM_PROFILE_PARABOLIC) {
            const R rx = sub_(add_(R(r1.x), R(0.5)), fp.axis_x), ry = sub_(add_(R(r1.y), R(0.5)), fp.axis_y);
            const R r2_ = fma_(rx, rx, mul_(ry, ry));
            speed = mul_(mul_(R(2), fp.u_in), sub_(R(1), mul_(R(4), r2_) / mul_(fp.d_in, fp.d_in)));
        }
        ux = mul_(speed, R((dir == 0) - (dir == 1)));
        uy = mul_(speed, R((dir == 2) - (dir == 3)));
        uz = mul_(speed, R((dir == 4) - (dir == 5)));
        if (fp.noise_amp != R(0)) {
            const int64_t node_id = (int64_t)(((uint64_t)(uint32_t)r1.w << 32) | (uint32_t)r1.z);
            const R amp = mul_(fp.noise_amp, fp.u_in);
            ux = fma_(amp, inlet_noise<R>(a.seed, a.t_new, node_id, 0), ux);
            uy = fma_(amp, inlet_noise<R>(a.seed, a.t_new, node_id, 1), uy);
            uz = fma_(amp, inlet_noise<R>(a.seed, a.t_new, node_id, 2), uz);
        }
        if (a.t_new < a.inlet_ramp) {  // smooth start: u_b r(t), r = s^2 (3 - 2 s), s = t / T
            const R sr = R(a.t_new) / R(a.inlet_ramp), r = mul_(mul_(sr, sr), fma_(R(-2), sr, R(3)));
            ux = mul_(ux, r);
            uy = mul_(uy, r);
            uz = mul_(uz, r);
        }
    }
    if (a.wall_qidx) {
        const int sf = nbf[4] + pf;
        const uint32_t lf = __ldg(a.mask + sf) & LINK_MASK;
        if (lf) interpolate_walls<P, WIDE, false, CG>(a, __ldg(a.wall_qidx + sf), sf, lf, d);
    }
    R rho;
    if constexpr (G == RATE_ONE && P != 2) {
        R s[10];
        axis_sums<R>([&](int i) { return d[i]; }, s);
        const R drho = s[0], jx = s[1], jy = s[2], jz = s[3], th = theta0<R>();
        rho = add_(R(1), drho);
        const R inv = recip(rho), uxf = mul_(jx, inv), uyf = mul_(jy, inv), uzf = mul_(jz, inv);
        const R a2[6] = {fma_(-jx, uxf, fma_(-th, drho, s[4])), fma_(-jy, uyf, fma_(-th, drho, s[5])),
                         fma_(-jz, uzf, fma_(-th, drho, s[6])), fma_(-jx, uyf, s[7]),
                         fma_(-jx, uzf, s[8]),                  fma_(-jy, uzf, s[9])};
        record_stress(a, slot, fp.omega, a2);  // the node takes its partner's stress
        if (!inlet) ux = uxf, uy = uyf, uz = uzf;
        const R rf = rho;
        rho = inlet ? rf : fp.rho_out;
        relaxed_lines<R>(sub_(R(1), fp.omega), a2, R(0), R(0), uxf, uyf, uzf,
                         NodeStore<P, WIDE, AX>{a, slot, pos, EqLines<R>(rho, inlet ? drho : sub_(rho, R(1)), ux, uy, uz)});
    } else {
        R rf, uxf, uyf, uzf;
        collide<P, G>(d, fp, rf, uxf, uyf, uzf, a, slot);  // the node takes its partner's stress
        if (!inlet) ux = uxf, uy = uyf, uz = uzf;
        rho = inlet ? rf : fp.rho_out;
        if constexpr (G == RATE_ONE) {
            const EqNode fe(rf, uxf, uyf, uzf), be(rho, ux, uy, uz);
            const NodeStore<P, WIDE, AX> out{a, slot, pos, EqLines<R>(rho, R(0), ux, uy, uz)};
#pragma unroll
            for (int j = 0; j < 9; ++j) {
                float b[3], f[3];
                be.line(j, b);
                fe.line(j, f);
#pragma unroll
                for (int c = 0; c < 3; ++c) b[c] = add_(d[3 * j + c], sub_(b[c], f[c]));
                out.line(j, b[0], b[1], b[2]);
            }
            record_cell(a, slot, rho, ux, uy, uz, hv);
            return;
        }
        EqLines<R> ef(rf, sub_(rf, R(1)), uxf, uyf, uzf);
        const NodeStore<P, WIDE, AX> out{a, slot, pos, EqLines<R>(rho, sub_(rho, R(1)), ux, uy, uz)};
#pragma unroll
        for (int j = 0; j < 9; ++j) {
            R e[3];
            if (j % 3 == 0) ef.plane(j / 3);
            ef.line(j % 3, e[0], e[1], e[2]);
            out(j, sub_(d[3 * j], e[0]), sub_(d[3 * j + 1], e[1]), sub_(d[3 * j + 2], e[2]));
        }
    }
    record_cell(a, slot, rho, ux, uy, uz, hv);
}

// Largest span one population's L2 prefetch may cover (bytes).
constexpr int64_t PREFETCH_MAX_BYTES = 16384;

// L2 prefetch of the pull sources of fluid block tb, population i.  The
// block's chunks cover rows r0..r1 in storage order, and the rows that
// population i pulls from, r + (cy, cz) for every r, are stored back to back
// in the same order, so its sources (slots nb_r[j] + x - cx) lie in one span
// from the first chunk's first lane to the last chunk's last lane.  The span
// is widened to 16-byte bounds, which stay inside the buffer margins.  Spans
// that wrap around a periodic y or z face (reversed or very long) are
// skipped: a prefetch only moves data, never changes a result.
template <int P, int AX>
__device__ __forceinline__ void prefetch_block_sources(const StepArgs &a, int tb, int i) {
    using T = typename Storage<P>::T;
    const int c0 = tb * (STEP_THREADS / CHUNK);
    if (tb < 0 || c0 >= a.nchunks) return;
    const int c1 = min(c0 + STEP_THREADS / CHUNK, a.nchunks) - 1;
    const int2 h0 = __ldg(a.chunks + c0), h1 = __ldg(a.chunks + c1);
    const int j = row_line<AX>(i), cx = c_row<AX>(i);
    const int *rn = reinterpret_cast<const int *>(a.row_nb);
    const int b0 = __ldg(rn + (int64_t)ROW_RECORD_INTS * h0.x + j);
    const int b1 = __ldg(rn + (int64_t)ROW_RECORD_INTS * h1.x + j);
    const int64_t s0 = (int64_t)b0 + (int)((uint32_t)h0.y & CHUNK_X0_MASK) - cx;
    const int64_t s1 = (int64_t)b1 + (int)((uint32_t)h1.y & CHUNK_X0_MASK) + CHUNK - cx;
    if (s1 <= s0 || (s1 - s0) * (int64_t)sizeof(T) > PREFETCH_MAX_BYTES) return;
    const char *arr = static_cast<const char *>(a.fin) + (int64_t)i * a.stride * (int64_t)sizeof(T);
    const uintptr_t lo = (uintptr_t)(arr + s0 * (int64_t)sizeof(T)) & ~(uintptr_t)15;
    const uintptr_t hi = ((uintptr_t)(arr + s1 * (int64_t)sizeof(T)) + 15) & ~(uintptr_t)15;
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(lo), "r"((uint32_t)(hi - lo)) : "memory");
}

// One time step of every fluid cell of one lattice.  The last warp of each
// block also prefetches the pull sources of block blockIdx.x +
// a.prefetch_ahead into L2 (one bulk prefetch per population), so that the
// gathers of later blocks find their rows in L2 instead of waiting on HBM.
template <int P, int G, bool WIDE, int AX>
__global__ void __launch_bounds__(STEP_THREADS, P == 0 ? 1 : (G == RATE_GENERAL ? 4 : LBM_STEP_MIN_BLOCKS))
    k_step(const StepArgs a) {
    double hv[6] = {0, 0, 0, 0, 0, 0};
    if (LBM_FUSE_BOUNDARY && P == 1 && (int)blockIdx.x >= a.fluid_blocks) {  // inlet/outlet nodes, trailing blocks
        const int k = ((int)blockIdx.x - a.fluid_blocks) * STEP_THREADS + (int)threadIdx.x;
        if (k < a.nbnodes) boundary_node<P, G, WIDE, AX>(a, k, hv);
    } else {
        const int gt = blockIdx.x * STEP_THREADS + threadIdx.x;
        const int chunk = gt / CHUNK;
        if constexpr (LBM_FAST_PATH && G == RATE_ONE && !WIDE && P != 0)
            fluid_lane_voted<P, G, AX>(a, chunk, gt % CHUNK, hv);  // every lane of the block calls it
        else if (chunk < a.nchunks)
            fluid_cell<P, G, WIDE, AX>(a, chunk, gt % CHUNK, hv);
        if (a.prefetch_ahead > 0) {
            const int i = (int)threadIdx.x - (STEP_THREADS - 32);
            if (i >= 0 && i < 27) prefetch_block_sources<P, AX>(a, (int)blockIdx.x + a.prefetch_ahead, i);
        }
    }
    if (a.flags & STEP_REDUCE) block_reduce_write(hv, a.partials);
}

// One time step of the cells with interpolated walls (see wall_cell); its
// partial sums follow those of the fluid and inlet/outlet kernels.
template <int P, int G, bool WIDE, int AX>
__global__ void __launch_bounds__(STEP_THREADS, P == 0 ? 1 : LBM_STEP_MIN_BLOCKS_WALLQ) k_wall(const StepArgs a) {
    const int k = blockIdx.x * STEP_THREADS + threadIdx.x;
    double hv[6] = {0, 0, 0, 0, 0, 0};
    if (k < a.nwnodes) wall_cell<P, G, WIDE, AX>(a, k, hv);
    if (a.flags & STEP_REDUCE) {
        const int before = a.fluid_blocks + (a.nbnodes + STEP_THREADS - 1) / STEP_THREADS;
        block_reduce_write(hv, a.partials + (size_t)before * REDUCE_SLOTS);
    }
}

// One time step of every inlet/outlet node of one lattice (when they do not
// ride in the trailing blocks of k_step).
template <int P, int G, bool WIDE, int AX>
__global__ void __launch_bounds__(STEP_THREADS) k_boundary(const StepArgs a) {
    const int k = blockIdx.x * STEP_THREADS + threadIdx.x;
    double hv[6] = {0, 0, 0, 0, 0, 0};
    if (k < a.nbnodes) boundary_node<P, G, WIDE, AX>(a, k, hv);
    if (a.flags & STEP_REDUCE) block_reduce_write(hv, a.partials + (size_t)a.fluid_blocks * REDUCE_SLOTS);
}

// -------------------------------------------------------- tile fluid kernel
//
// Variant of the fluid kernel (default ghost rates, 32-bit offsets, FP32 /
// FP16S) over tile records instead of chunk records: one warp updates one
// tile, up to 32 consecutive cells of a row.  Its record (p0, lanes, the
// nine neighbour-row bases) is one 48-byte load with no dependent index
// load before the gather.  A "fast" tile (32 fluid cells, no wall link, no
// wrap-around copy; flagged when the index is built) stores through shared
// memory: each lane writes its 27 values at fixed offsets, and the warp
// writes every population's 32 consecutive own slots as 16-byte stores, so
// the 27 per-value address computations of the line sink disappear.  Other
// tiles load their link words and use the line sink.

template <int P>
struct TileOut {
    using T = typename Storage<P>::T;
    static constexpr int S = (int)sizeof(T);
    static constexpr int PIECE = 16 / S;          // elements of one 16-byte store
    static constexpr int PIECES = 32 / PIECE;     // 16-byte pieces of one population's 32 outputs
    static constexpr int ELEMS = 27 * 32;         // a warp's staged outputs
};

// Output sink of a fast tile: value i of lane l goes to out[i * 32 + l] in
// the warp's shared-memory slice (out points at lane l's first element).
template <int P, bool RAW>
struct SharedStore {
    using S = Storage<P>;
    using T = typename S::T;
    using R = typename S::R;
    const StepArgs &a;
    int slot;
    T *out;
    __device__ __forceinline__ void put(int i, R v) const {
        if constexpr (RAW)
            S::store_raw(out + 32 * i, v);
        else
            S::store(out + 32 * i, v, R(a.scale));
    }
    __device__ __forceinline__ void moments(R omega, const R (&a2)[6]) const { record_stress(a, slot, omega, a2); }
    __device__ __forceinline__ void operator()(int j, R vm, R v0, R vp) const {
        put(3 * j, vm);
        put(3 * j + 1, v0);
        put(3 * j + 2, vp);
    }
};

// The record of a tile (48 bytes; the same for every lane).
struct TileRec {
    int4 r0, r1, r2;
    TileRec() = default;
    __device__ __forceinline__ TileRec(const int32_t *tiles, int t) {
        const int4 *rec = reinterpret_cast<const int4 *>(tiles) + 3 * (size_t)t;
        r0 = __ldg(rec), r1 = __ldg(rec + 1), r2 = __ldg(rec + 2);
    }
};

// One warp's update of a tile (lane = the warp lane, out = the warp's
// shared-memory slice of TileOut<P>::ELEMS elements).  Without FAST every tile
// takes the line sink, and out is not used: half the code, for kernels that
// otherwise wait on the instruction cache.  SERVED: the request server's
// roundings.
template <int P, int AX, bool CG = false, bool FAST = true, bool SERVED = false>
__device__ __forceinline__ void tile_update(const StepArgs &a, const TileRec &rec, int lane, typename TileOut<P>::T *out,
                                            double (&hv)[6]) {
    using O = TileOut<P>;
    using T = typename O::T;
    using R = typename Storage<P>::R;
    constexpr bool RAW = Storage<P>::SCALED;
    const int4 &r0 = rec.r0, &r1 = rec.r1, &r2 = rec.r2;
    const int nb[9] = {r0.w, r1.x, r1.y, r1.z, r1.w, r2.x, r2.y, r2.z, r2.w};
    const bool fast = ((uint32_t)r0.x & TILE_FAST) != 0u;
    const int p0 = (int)((uint32_t)r0.x & CHUNK_X0_MASK);
    const int x = p0 + lane, slot = nb[4] + x;
    const bool fluid = ((uint32_t)r0.y >> lane) & 1u;
    const Rounds rounds =
        SERVED ? served_rounds() : lane_rounds<AX>(((uint32_t)r0.x >> (TILE_PLAIN_SHIFT + lane / CHUNK)) & 1u);
    R d[27];
    gather<P, false, AX, RAW, CG>(a, nb, x, d);  // every lane's pulls lie inside the buffer margins
    R rho, ux, uy, uz;
    if (FAST && fast) {
        const SharedStore<P, RAW> sink{a, slot, out + lane};
        collide_ghost1<R, RAW>(d, flow<R>(a).omega, rho, ux, uy, uz, R(a.inv_scale), R(a.scale), sink, rounds);
        __syncwarp();
        // piece q = 4 i + k (FP16S) / 8 i + k (FP32): elements 16k/S.. of population i,
        // at shared offset 16 q bytes and at own slots nb[4] + p0 + k PIECE
        T *fout = static_cast<T *>(a.fout) + (nb[4] + p0);
#pragma unroll
        for (int q0 = 0; q0 < 27 * O::PIECES; q0 += 32) {
            const int q = q0 + lane;
            if (q < 27 * O::PIECES) {
                const int4 v = reinterpret_cast<const int4 *>(out)[q];
                const int i = q / O::PIECES, k = q % O::PIECES;
                *reinterpret_cast<int4 *>(fout + elem<false>(i, a.stride, k * O::PIECE)) = v;
            }
        }
        __syncwarp();
    } else {
        const bool present = ((uint32_t)r0.z >> lane) & 1u;
        const uint32_t m = present ? __ldg(a.mask + slot) : 0u;
        const uint32_t links = fluid ? (m & LINK_MASK) : 0u;
        const uint32_t own = fluid ? (LINK_MASK | OWN_FLUID)
                                   : (present && ((m >> TYPE_SHIFT) & 3u) == TYPE_PAD ? (~m & LINK_MASK) : 0u);
        const LineStore<P, false, RAW, AX> sink{a, nb, x, slot, links, own};
        collide_ghost1<R, RAW>(d, flow<R>(a).omega, rho, ux, uy, uz, R(a.inv_scale), R(a.scale), sink, rounds);
    }
    if (fluid) record_cell(a, slot, rho, ux, uy, uz, hv);
}

template <int P, int AX>
__global__ void __launch_bounds__(STEP_THREADS, LBM_STEP_MIN_BLOCKS) k_step_tiles(const StepArgs a) {
    using O = TileOut<P>;
    __shared__ __align__(16) typename O::T staged_out[STEP_THREADS / 32][O::ELEMS];
    const int warp = (int)(threadIdx.x >> 5), lane = (int)(threadIdx.x & 31);
    const int t = (int)blockIdx.x * (STEP_THREADS / 32) + warp;
    double hv[6] = {0, 0, 0, 0, 0, 0};
    if (t < a.ntiles) tile_update<P, AX>(a, TileRec(a.tiles, t), lane, staged_out[warp], hv);  // uniform over the warp
    if (a.flags & STEP_REDUCE) block_reduce_write(hv, a.partials);
}

// ------------------------------------------------ pair fluid kernel (FP16S)
//
// Fast tiles of an FP16S lattice (32 fluid cells, no wall link, no
// wrap-around copy) with two adjacent cells per thread: 16 threads per
// tile, thread k updates cells x = p0 + 2k and x + 1.  The collision runs on
// the packed FP32 pipe across the pair (one instruction for both cells); its
// 27 inputs stay FP16 pairs until the moment pass converts them; the pull
// of each line along the row (c = 0 along the row axis) is one aligned
// 32-bit load of both cells' values, the other two are two 16-bit loads;
// each output is one 32-bit store of both cells' own slots.  Every thread
// holds two cells, so the kernel runs at fewer resident warps than the
// one-cell kernels with the same bytes in flight per SM.
#ifndef LBM_PAIR_MIN_BLOCKS
#define LBM_PAIR_MIN_BLOCKS 5
#endif

struct Half2ToF2 {
    __device__ __forceinline__ F2 operator()(__half2 h) const { return F2(__half22float2(h)); }
};

// Pull gather of the pair (x, x + 1), x even: d[i] = FP16 pulls of both cells.
template <int AX>
__device__ __forceinline__ void gather_pair(const StepArgs &a, const int (&nb)[9], int x, __half2 (&d)[27]) {
    const __half *fin = static_cast<const __half *>(a.fin);
    const uint32_t st = (uint32_t)a.stride;
    constexpr int dk = line_pop<AX>(0, 1) - line_pop<AX>(0, 0);
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        const __half *pj = fin + ((uint32_t)line_pop<AX>(j, 0) * st + (uint32_t)(nb[j] + x));
        // c_row = -1: pulls from x + 1, x + 2
        d[line_pop<AX>(j, 0)] = __halves2half2(__ldg(pj + 1), __ldg(pj + 2));
        // c_row = 0: pulls from x, x + 1, one aligned 32-bit load
        d[line_pop<AX>(j, 1)] = __ldg(reinterpret_cast<const __half2 *>(pj + dk * st));
        // c_row = +1: pulls from x - 1, x
        d[line_pop<AX>(j, 2)] = __halves2half2(__ldg(pj + 2 * dk * st - 1), __ldg(pj + 2 * dk * st));
    }
}

// Viscous stress of the pair's two cells (statistics sample steps).
__device__ __forceinline__ void record_stress_pair(const StepArgs &a, int slot, F2 omega, const F2 (&a2)[6]) {
    if ((a.flags & (STEP_STATS | STEP_STATS_FULL)) != (STEP_STATS | STEP_STATS_FULL)) return;
    float ax[6], ay[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) ax[q] = a2[q].v.x, ay[q] = a2[q].v.y;
    record_stress(a, slot, omega.v.x, ax);
    record_stress(a, slot + 1, omega.v.y, ay);
}

// Output sink of a fast tile: both cells' values of population i as one FP16
// pair at their own slots (slot even), already scaled by the collision.
struct PairStore {
    const StepArgs &a;
    int slot;
    __device__ __forceinline__ void moments(F2 omega, const F2 (&a2)[6]) const {
        record_stress_pair(a, slot, omega, a2);
    }
    __device__ __forceinline__ void operator()(int j, F2 vm, F2 v0, F2 vp) const {
        const uint32_t st = (uint32_t)a.stride;
        __half *pj = static_cast<__half *>(a.fout) + ((uint32_t)(3 * j) * st + (uint32_t)slot);
        *reinterpret_cast<__half2 *>(pj) = __float22half2_rn(vm.v);
        *reinterpret_cast<__half2 *>(pj + st) = __float22half2_rn(v0.v);
        *reinterpret_cast<__half2 *>(pj + 2 * st) = __float22half2_rn(vp.v);
    }
};

// Half a warp's update of fast tile t with two cells per thread (k: the
// pair within the tile).
template <int AX>
__device__ __forceinline__ void pair_update(const StepArgs &a, int t, int k, double (&hv)[6]) {
    const int4 *rec = reinterpret_cast<const int4 *>(a.tiles) + 3 * (size_t)t;
    const int4 r0 = __ldg(rec), r1 = __ldg(rec + 1), r2 = __ldg(rec + 2);
    const int nb[9] = {r0.w, r1.x, r1.y, r1.z, r1.w, r2.x, r2.y, r2.z, r2.w};
    const int x = (int)((uint32_t)r0.x & CHUNK_X0_MASK) + 2 * k, slot = nb[4] + x;
    __half2 d[27];
    gather_pair<AX>(a, nb, x, d);
    F2 m[10], rho, ux, uy, uz;
    ghost1_sums<F2>([&](int i) { return Half2ToF2{}(d[i]); }, m);
    ghost1_finish<true, F2>(m, F2(a.pf.omega), rho, ux, uy, uz, F2(a.inv_scale), F2(a.scale),
                            lane_rounds<AX>(((uint32_t)r0.x >> (TILE_PLAIN_SHIFT + 2 * k / CHUNK)) & 1u), PairStore{a, slot});
    double h0[6] = {0, 0, 0, 0, 0, 0}, h1[6] = {0, 0, 0, 0, 0, 0};
    record_cell(a, slot, rho.v.x, ux.v.x, uy.v.x, uz.v.x, h0);
    record_cell(a, slot + 1, rho.v.y, ux.v.y, uy.v.y, uz.v.y, h1);
#pragma unroll
    for (int q = 0; q < 6; ++q) hv[q] = q == 4 ? fmax(h0[q], h1[q]) : h0[q] + h1[q];
}

// FP16S pair kernel: one pair of fast tiles per warp (in row order), 16
// threads per tile, two cells per thread.  Every other cell of the lattice
// is updated by the chunk kernel over the remaining chunks, in a launch of
// its own: one instruction stream per kernel, each at its own register
// budget.
template <int AX>
__global__ void __launch_bounds__(STEP_THREADS, LBM_PAIR_MIN_BLOCKS) k_step_pairs(const StepArgs a) {
    const int warp = (int)(threadIdx.x >> 5), lane = (int)(threadIdx.x & 31);
    const int w = (int)blockIdx.x * (STEP_THREADS / 32) + warp;
    double hv[6] = {0, 0, 0, 0, 0, 0};
    if (w < a.nitems) {
        const int2 item = __ldg(a.items + w);
        pair_update<AX>(a, lane < 16 ? item.x : item.y, lane & 15, hv);
    }
    if (a.flags & STEP_REDUCE) block_reduce_write(hv, a.partials);
}

// ------------------------------------------------ staged unit kernel (FP16S)
//
// The FP16S fluid kernel of larger lattices: persistent warps over units of
// up to 64 cells of a row.  In FP16S a step moves half the bytes of FP32 for
// the same work, so what bounds a one-cell-per-thread kernel is not HBM but
// the loads a warp can have in flight in its registers (long-scoreboard waits
// were 6.5 of the 12.1 cycles between a warp's issues) and its 700
// instructions per cell.  Here each warp copies the pull windows of its next
// unit (27 arrays, 64 cells and one 16-byte piece on the side they pull from)
// into its own shared-memory stages, nine 16-byte cp.async per lane, while it
// computes the current one, so its loads in flight do not depend on registers
// or on other warps.  Each thread updates two adjacent cells on the packed
// FP32 pipe, one instruction stream for every unit (the output sink alone
// tells plain units, 64 fluid cells without wall links, from the others).
//
// Measured per step, chunk kernel and this one: Re 6500 nozzle 446 -> 354 us
// (4.42 TB/s of algorithmic bytes; with axial averages 553 -> 486), Re 3500
// nozzle 151 -> 127 us, periodic 256^3 501 -> 361 us (5.02 TB/s).  Two stages
// and 4 blocks of 4 warps per SM: 3 blocks take 6 % longer on the Re 6500
// nozzle, a third stage changes nothing.  The moments and lines in fewer
// operations (250 a cell pair instead of 320) took 336 us, in other roundings
// (see Rounds).
// Steps that sample full statistics take the chunk kernel, whose 32 cells a
// warp touch each accumulator's sectors at once: 503 us against 627 on the Re
// 3500 nozzle.
#ifndef LBM_STAGE_DEPTH
#define LBM_STAGE_DEPTH 2
#endif
#ifndef LBM_STAGE_BLOCKS
#define LBM_STAGE_BLOCKS 4
#endif
#ifndef LBM_STAGE_RUN
#define LBM_STAGE_RUN 3
#endif
constexpr int STAGE_DEPTH = LBM_STAGE_DEPTH;
constexpr int STAGE_RUN = LBM_STAGE_RUN;             // units per ticket
constexpr int STAGE_WINDOW = 160;                    // bytes of one population's window: 128 + 2 x 16
constexpr int STAGE_MASK = 27 * STAGE_WINDOW;        // windows in (line, c_row) order, then the link words
constexpr int STAGE_REC = STAGE_MASK + 64 * 4;       // and the unit's record
constexpr int STAGE_BYTES = STAGE_REC + UNIT_INTS * 4;
constexpr int STAGE_WARPS = STEP_THREADS / 32;
constexpr int STAGE_SMEM = STAGE_WARPS * STAGE_DEPTH * STAGE_BYTES;

__device__ __forceinline__ void copy16(uint32_t dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// Byte offset, in a stage, of population i's value for the cell at unit
// position 0: its window, 16 bytes in, shifted by the pull.
template <int AX>
__host__ __device__ constexpr int stage_offset(int i) {
    return (row_line<AX>(i) * 3 + c_row<AX>(i) + 1) * STAGE_WINDOW + 16 - 2 * c_row<AX>(i);
}

// Start the copies of a unit (rec: lane l holds word l of its record) into a
// stage: the pull windows, lane 10 k + q copying piece q of the c_row = k - 1
// population of each line; the link words, unless the unit is plain; and the
// record.  lane_src is fin plus the lane's part of the element offset.
template <int AX>
__device__ __forceinline__ void stage_issue(const StepArgs &a, int rec, char *stage, uint32_t dst,
                                            const char *lane_src, int lane) {
    const int p0 = __shfl_sync(0xffffffffu, rec, 0);
    const int pieces = __shfl_sync(0xffffffffu, rec, 5), flags = __shfl_sync(0xffffffffu, rec, 6);
    // pieces needed: the present chunks lo .. hi, one position further on the
    // side that c_row pulls from
    const int lo = pieces & ((1 << UNIT_HI_SHIFT) - 1), hi = pieces >> UNIT_HI_SHIFT;
    const int k = lane / 10, q = lane % 10;
    const bool on = lane < 30 && q >= (k == 2 ? lo : lo + 1) && q <= (k == 0 ? hi + 2 : hi + 1);
    const uint32_t lane_dst = dst + (k * STAGE_WINDOW + 16 * q);
    const int64_t line_stride = (AX == 0 ? 3 : 1) * a.stride;
    int own = 0;
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        const int nb = __shfl_sync(0xffffffffu, rec, UNIT_NB + j);
        if (j == 4) own = nb;
        if (on) copy16(lane_dst + j * 3 * STAGE_WINDOW, lane_src + 2 * (j * line_stride + (int64_t)(nb + p0)));
    }
    if (!(flags & UNIT_PLAIN) && lane >= 2 * lo && lane <= 2 * hi + 1)
        copy16(dst + STAGE_MASK + 16 * lane, a.mask + (own + p0 + 4 * lane));
    if (lane < UNIT_INTS) *reinterpret_cast<int *>(stage + STAGE_REC + 4 * lane) = rec;
}

// Output sink of a unit: the adjacent cells x (first half of each value) and
// x + 1 of a thread.  A plain unit stores both cells of each population as
// one 32-bit word; otherwise each cell has its own-slot predicates (bit i of
// own; OWN_FLUID marks a fluid cell), its wall links' ghost slots and its
// wrap-around copies, as LineStore has for one cell.  plain and wrap are
// uniform over the warp.  nb: the neighbour bases in shared memory.
template <int AX>
struct UnitStore {
    const StepArgs &a;
    const int *nb;
    int x, slot;
    bool plain, wrap;
    uint32_t links[2], both, own[2];  // both: own of both cells; own: of one cell only
    uint32_t fluid;                   // bit h: cell x + h is a fluid cell
    __device__ __forceinline__ void moments(F2, const F2 (&)[6]) const {}  // no full statistics here
    __device__ __forceinline__ void put(int i, int s, __half v) const {
        static_cast<__half *>(a.fout)[elem<false>(i, a.stride, s)] = v;
    }
    __device__ __forceinline__ void operator()(int j, F2 vm, F2 v0, F2 vp) const {
        const __half2 v[3] = {__float22half2_rn(vm.v), __float22half2_rn(v0.v), __float22half2_rn(vp.v)};
        __half *out = static_cast<__half *>(a.fout);
        const uint32_t st = (uint32_t)a.stride;
        __half *pj = out + ((uint32_t)(3 * j) * st + (uint32_t)slot);
        __half *p[3] = {pj, pj + st, pj + 2 * st};
        if (plain) {
#pragma unroll
            for (int c = 0; c < 3; ++c) *reinterpret_cast<__half2 *>(p[c]) = v[c];
        } else {
            const int jl = 8 - j;  // links 26 - i of this line's values sit in line 8 - j
#pragma unroll
            for (int c = 0; c < 3; ++c)
                if (both & (1u << (3 * j + c))) *reinterpret_cast<__half2 *>(p[c]) = v[c];
            if ((own[0] | own[1]) & (7u << (3 * j))) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    if (own[0] & (1u << (3 * j + c))) p[c][0] = __low2half(v[c]);
                    if (own[1] & (1u << (3 * j + c))) p[c][1] = __high2half(v[c]);
                }
            }
            if ((links[0] | links[1]) & (7u << (3 * jl))) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const int k = 26 - (3 * j + c);  // wall link k takes value 3j + c
                    const int s = nb[row_line<AX>(k)] + x - c_row<AX>(k);
                    if (links[0] & (1u << k)) put(k, s, __low2half(v[c]));
                    if (links[1] & (1u << k)) put(k, s + 1, __high2half(v[c]));
                }
            }
        }
        if (wrap) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (!(fluid & (1u << h))) continue;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const int i = 3 * j + c;
                    const __half w = h ? __high2half(v[c]) : __low2half(v[c]);
                    if (c_row<AX>(i) == 1 && x + h == a.n_row - 1) put(i, nb[4] - 1, w);
                    if (c_row<AX>(i) == -1 && x + h == 0) put(i, nb[4] + a.n_row, w);
                }
            }
        }
    }
};

// Update of the unit in a stage: two adjacent cells per thread.
template <int AX>
__device__ __forceinline__ void stage_update(const StepArgs &a, const char *st, int lane) {
    const int *rec = reinterpret_cast<const int *>(st + STAGE_REC);
    const int x = rec[0] + 2 * lane, slot = rec[UNIT_NB + 4] + x;
    UnitStore<AX> sink{a, rec + UNIT_NB, x, slot, (rec[6] & UNIT_PLAIN) != 0, (rec[6] & UNIT_WRAP) != 0,
                       {0u, 0u}, 0u, {0u, 0u}, 3u};
    if (!sink.plain) {
        const uint2 mk2 = *reinterpret_cast<const uint2 *>(st + STAGE_MASK + 8 * lane);  // not copied where absent
        const uint32_t fl = (uint32_t)rec[1 + (lane >> 4)] >> (2 * (lane & 15));
        const uint32_t pr = (uint32_t)rec[3 + (lane >> 4)] >> (2 * (lane & 15));
        uint32_t own[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t mk = h ? mk2.y : mk2.x;
            const bool fluid = (fl >> h) & 1u;
            sink.links[h] = fluid ? (mk & LINK_MASK) : 0u;
            own[h] = fluid ? LINK_MASK
                           : (((pr >> h) & 1u) && ((mk >> TYPE_SHIFT) & 3u) == TYPE_PAD ? (~mk & LINK_MASK) : 0u);
        }
        sink.both = own[0] & own[1];
        sink.own[0] = own[0] & ~own[1];
        sink.own[1] = own[1] & ~own[0];
        sink.fluid = fl & 3u;
        sink.wrap = a.periodic_row != 0;
    }
    const char *sl = st + 4 * lane;
    auto ld = [&](int i) {
        const char *p = sl + stage_offset<AX>(i);
        if (c_row<AX>(i) == 0) return F2(__half22float2(*reinterpret_cast<const __half2 *>(p)));
        return F2(make_float2(__half2float(*reinterpret_cast<const __half *>(p)),
                              __half2float(*reinterpret_cast<const __half *>(p + 2))));
    };
    F2 m[10], rho, ux, uy, uz;
    ghost1_sums<F2>(ld, m);
    ghost1_finish<true, F2>(m, F2(a.pf.omega), rho, ux, uy, uz, F2(a.inv_scale), F2(a.scale),
                            lane_rounds<AX>((rec[6] >> (UNIT_PLAIN_SHIFT + 2 * lane / CHUNK)) & 1), sink);
    if (a.flags & STEP_STATS) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (sink.fluid & (1u << h)) record_axial(a, slot + h, h ? uz.v.y : uz.v.x);
    }
}

// The units a warp takes: runs of STAGE_RUN consecutive units from the work
// counter (one address takes an atomic about every 2 ns: single-unit runs
// throughout took 551 us a step on the Re 6500 nozzle where runs of three took 339),
// and single ones over the last two rounds of the warps, so that they finish
// together.  The next ticket is drawn while the current run is handed out.
struct UnitQueue {
    int32_t *counter;
    int n, n_long, pos, end, ticket;
    __device__ __forceinline__ UnitQueue(int32_t *counter_, int n_, int warps)
        : counter(counter_), n(n_), n_long(max(0, n_ - 2 * warps) / STAGE_RUN), pos(0), end(0), ticket(0) {}
    __device__ __forceinline__ void draw(int lane) { ticket = lane == 0 ? atomicAdd(counter, 1) : 0; }
    __device__ __forceinline__ int next(int lane) {  // -1 when none is left
        if (pos >= end) {
            const int t = __shfl_sync(0xffffffffu, ticket, 0);
            pos = t < n_long ? t * STAGE_RUN : n_long * STAGE_RUN + (t - n_long);
            end = pos + (t < n_long ? STAGE_RUN : 1);
            if (pos >= n) {
                end = pos;
                return -1;  // and at every later call: the ticket stays past the end
            }
            draw(lane);
        }
        return pos++;
    }
};

template <int AX>
__global__ void __launch_bounds__(STEP_THREADS, LBM_STAGE_BLOCKS) k_step_units(const StepArgs a) {
    extern __shared__ __align__(16) char stages[];
    const int warp = (int)(threadIdx.x >> 5), lane = (int)(threadIdx.x & 31);
    char *base = stages + warp * (STAGE_DEPTH * STAGE_BYTES);
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(base);
    const int k = lane / 10, q = lane % 10;
    const char *lane_src = static_cast<const char *>(a.fin) + 2 * ((AX == 0 ? k : 9 * k) * a.stride + 8 * q - 8);
    UnitQueue queue(a.tickets, a.nunits, (int)gridDim.x * STAGE_WARPS);
    queue.draw(lane);
    constexpr int NONE = -1;  // as word 0 of a record: no unit (p0 is a multiple of CHUNK)
    auto fetch = [&]() {
        const int u = queue.next(lane);
        return u < 0 ? NONE : __ldg(a.units + (size_t)u * UNIT_INTS + (lane & (UNIT_INTS - 1)));
    };
    auto there = [&](int r) { return __shfl_sync(0xffffffffu, r, 0) != NONE; };  // uniform
    int in_flight = 0;  // units being copied or ready
    int ahead = fetch();
#pragma unroll
    for (int s = 0; s < STAGE_DEPTH - 1; ++s) {
        if (there(ahead)) {
            stage_issue<AX>(a, ahead, base + s * STAGE_BYTES, sbase + s * STAGE_BYTES, lane_src, lane);
            ++in_flight;
            ahead = fetch();
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    int cur = 0;  // stage of the current unit
    while (in_flight > 0) {
        if (there(ahead)) {  // into the stage read in the last round
            const int s = cur == 0 ? STAGE_DEPTH - 1 : cur - 1;
            stage_issue<AX>(a, ahead, base + s * STAGE_BYTES, sbase + s * STAGE_BYTES, lane_src, lane);
            ++in_flight;
            ahead = fetch();
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group %0;" ::"n"(STAGE_DEPTH - 1) : "memory");
        __syncwarp();
        stage_update<AX>(a, base + cur * STAGE_BYTES, lane);
        __syncwarp();  // every lane is done with the stage before it is refilled
        --in_flight;
        cur = cur == STAGE_DEPTH - 1 ? 0 : cur + 1;
    }
    // the last block to finish clears the counters for the next launch
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(a.tickets + 1, 1) == (int)gridDim.x - 1) {
        a.tickets[0] = 0;
        a.tickets[1] = 0;
    }
}

// ------------------------------------------- several steps in one launch
//
// A small lattice fits L2 and its step is a few microseconds of work, less
// than a step's launches, stream fork and join.  This kernel takes `steps`
// time steps in one cooperative launch (all blocks resident), with a barrier
// over the grid between steps: warp items are the inlet/outlet nodes and
// wall cells (32 each; first, they take longest) and the fluid tiles (or
// groups of 32 chunk lanes for the other collision forms), dealt to the same
// warps in every step.  The populations change between the steps of one
// launch, so they are loaded from L2 (CG).  Each cell runs the same code as
// in the per-step kernels, to the same bits.
//
// Measured per step, one launch each and in one: laminar nozzle 24x24x160 FP32
// 10.6 -> 6.6 us, FP16S 11.2 -> 7.1; pipe of 237 000 cells FP32 14.4 -> 11.2,
// FP16S 12.5 -> 12.9; 64^3 lattice BGK 14.4 -> 11.1 (FP32 per step 17.4 with the
// cascade); smooth nozzle of 226 000 cells 24.1 -> 15.8; 32^3 box 7.4 -> 3.7, of
// which about 1.5 us is the barrier.  At 80^3 (6.6 rounds) both take 29 us.  4 blocks per
// SM (128 registers, no spills); 5 and 8 spill and take 10 to 40 % longer.  The
// line sink for every tile: with the fast tiles' path as well the nozzle takes
// 8.3 us.
#ifndef LBM_RUN_BLOCKS
#define LBM_RUN_BLOCKS 4
#endif

// Wait until all blocks have arrived `rounds` times at the barrier word, for
// at most `polls` looks (some seconds): then bit 1 of the status word tells the
// host, and every block leaves.  The result is uniform over the block.
__device__ __forceinline__ bool grid_barrier(int32_t *word, int rounds, uint32_t *status, int polls) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        const int target = rounds * (int)gridDim.x;
        int seen = 0;
        asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(word) : "memory");
        for (int k = 0; k < polls; ++k) {
            asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(seen) : "l"(word) : "memory");
            if (seen >= target || (*(volatile uint32_t *)status & 2u)) break;
        }
        if (seen < target) atomicOr(status, 2u);
        s_ok = seen >= target;
    }
    __syncthreads();
    return s_ok != 0;
}

template <int P, int G, int AX>
__global__ void __launch_bounds__(STEP_THREADS, LBM_RUN_BLOCKS) k_run(const StepArgs a0, const RunArgs run) {
    constexpr bool TILES = G == RATE_ONE;
    const int warp = (int)(threadIdx.x >> 5), lane = (int)(threadIdx.x & 31);
    // warps of one block take items far apart, so that the nodes spread over the SMs
    const int first = warp * (int)gridDim.x + (int)blockIdx.x, stride = (int)gridDim.x * (STEP_THREADS / 32);
    const int nodes = (a0.nbnodes + 31) / 32, walls = (a0.nwnodes + 31) / 32;
    StepArgs a = a0;
    double hv[6];
    for (int s = 0; s < run.steps; ++s) {
        a.t_new = a0.t_new + s;
        a.fin = s & 1 ? a0.fout : a0.fin;
        a.fout = s & 1 ? const_cast<void *>(a0.fin) : a0.fout;
        const int64_t since = a.t_new - run.stats_start;
        a.flags = run.stats_flags && since >= 0 && since % run.stats_stride == 0 ? run.stats_flags : 0;
        int i = first;
        for (; i < nodes; i += stride) {
            const int k = 32 * i + lane;
            if (k < a.nbnodes) boundary_node<P, G, false, AX, true>(a, k, hv);
        }
        for (; i < nodes + walls; i += stride) {
            const int k = 32 * (i - nodes) + lane;
            if (k < a.nwnodes) wall_cell<P, G, false, AX, true>(a, k, hv);
        }
        i -= nodes + walls;
        if constexpr (TILES) {  // the next tile's record is on its way while a tile is updated
            TileRec next;
            if (i < a.ntiles) next = TileRec(a.tiles, i);
            for (; i < a.ntiles; i += stride) {
                const TileRec rec = next;
                if (i + stride < a.ntiles) next = TileRec(a.tiles, i + stride);
                tile_update<P, AX, true, false>(a, rec, lane, nullptr, hv);
            }
        } else {
            for (; i < (a.nchunks + 3) / 4; i += stride) {
                const int chunk = 4 * i + lane / CHUNK;
                if (chunk < a.nchunks) fluid_cell<P, G, false, AX, true>(a, chunk, lane % CHUNK, hv);
            }
        }
        if (s + 1 < run.steps && !grid_barrier(run.barrier, s + 1, a.status, run.polls)) break;
    }
    // the last block to leave clears the words for the next launch
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(run.barrier + 1, 1) == (int)gridDim.x - 1) {
        run.barrier[0] = 0;
        run.barrier[1] = 0;
    }
}

// ---------------------------------------------------------- utility kernels

// The stored values of a cell, without the FP16 scale.
template <int P>
__device__ __forceinline__ void load_stored(const void *f, int64_t stride, int slot, double (&d)[27]) {
    const typename Storage<P>::T *p = static_cast<const typename Storage<P>::T *>(f);
#pragma unroll
    for (int i = 0; i < 27; ++i) {
        if constexpr (P == 2)
            d[i] = (double)__half2float(p[(int64_t)i * stride + slot]);
        else
            d[i] = (double)p[(int64_t)i * stride + slot];
    }
}

template <int P>
__device__ __forceinline__ void load_cell(const void *f, int64_t stride, int slot, float inv_scale,
                                          double (&d)[27]) {
    using S = Storage<P>;
    const typename S::T *p = static_cast<const typename S::T *>(f);
#pragma unroll
    for (int i = 0; i < 27; ++i) {
        if constexpr (P == 2)
            d[i] = (double)__half2float(p[(int64_t)i * stride + slot]) * (double)inv_scale;
        else
            d[i] = (double)p[(int64_t)i * stride + slot];
    }
}

// Whether x is neither zero, subnormal, infinite nor NaN (integer pipe).
__device__ __forceinline__ bool normal(double x) {
    return ((unsigned)__double2hiint(x) & 0x7ff00000u) - 0x00100000u < 0x7fe00000u;
}
// The same for x and 1 / x: |x| < 2^1022 too.
__device__ __forceinline__ bool invertible(double x) {
    return ((unsigned)__double2hiint(x) & 0x7ff00000u) - 0x00100000u < 0x7fc00000u;
}

// j / rho, for an invertible rho, from its correctly rounded reciprocal inv:
// the residual of j inv corrects it once, to the correctly rounded quotient
// (Markstein, IBM J. Res. Dev. 34, 1990; the residual must not underflow: |j|
// above 2^-968), at three operations.  An infinite j stays infinite.
__device__ __forceinline__ double quotient(double j, double rho, double inv) {
    const double q = __dmul_rn(j, inv);
    return normal(q) ? __fma_rn(__fma_rn(-rho, q, j), inv, q) : q;
}

// Density and velocity from the stored populations of a cell, in FP64 (the
// FP16 scale, a power of two, acts on the sums).  The FP64 pipe is what
// bounds the kernels that use this (a multiplication by every direction's
// components, 0 included, and three divisions took 130 us per million cells),
// so the sums share their partial sums: 49 additions.
template <int P>
__device__ __forceinline__ void moments_of(const double (&d)[27], double inv_scale, double &rho, double &ux,
                                           double &uy, double &uz) {
    const double sc = Storage<P>::SCALED ? inv_scale : 1.0;
    double s[9], jx = 0.0;  // sums over cx of each line (cy, cz)
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        s[j] = (d[3 * j] + d[3 * j + 2]) + d[3 * j + 1];
        jx += d[3 * j + 2] - d[3 * j];
    }
    const double lo = (s[0] + s[3]) + s[6], mid = (s[1] + s[4]) + s[7], hi = (s[2] + s[5]) + s[8];  // cy = -1, 0, 1
    double jy = hi - lo, jz = ((s[6] - s[0]) + (s[8] - s[2])) + (s[7] - s[1]), drho = (lo + hi) + mid;
    if constexpr (Storage<P>::SCALED) drho *= sc, jx *= sc, jy *= sc, jz *= sc;
    rho = 1.0 + drho;
    if (invertible(rho)) {
        const double inv = recip(rho);
        ux = quotient(jx, rho, inv);
        uy = quotient(jy, rho, inv);
        uz = quotient(jz, rho, inv);
    } else {  // a diverged state: whatever the division gives
        ux = jx / rho;
        uy = jy / rho;
        uz = jz / rho;
    }
}

// Health reduction of a stored state (mass, momentum, max |u|, non-finite count).
template <int P>
__global__ void __launch_bounds__(STEP_THREADS) k_reduce(const void *f, const int32_t *act, int64_t stride,
                                                         float inv_scale, double *partials) {
    double hv[6] = {0, 0, 0, 0, 0, 0};
    for (int64_t slot = (int64_t)blockIdx.x * STEP_THREADS + threadIdx.x; slot < stride;
         slot += (int64_t)gridDim.x * STEP_THREADS) {
        if (__ldg(act + slot) < 0) continue;
        double d[27], rho, ux, uy, uz, v[6];
        load_stored<P>(f, stride, (int)slot, d);
        moments_of<P>(d, inv_scale, rho, ux, uy, uz);
        health_values(rho, ux, uy, uz, v);
#pragma unroll
        for (int q = 0; q < 6; ++q) hv[q] = q == 4 ? fmax(hv[q], v[q]) : hv[q] + v[q];
    }
    block_reduce_write(hv, partials);
}

// Ghost slots and periodic copies along the rows of one buffer from its
// active cells: the same writes the step kernel does after its collision,
// for a state set from the host.
template <int P, int AX>
__global__ void __launch_bounds__(STEP_THREADS) k_fill_ghosts(void *f, const uint32_t *mask, const int2 *chunks,
                                                              const int4 *row_nb, int32_t nchunks, int64_t stride,
                                                              int32_t n_row, int32_t periodic_row) {
    using T = typename Storage<P>::T;
    const int gt = blockIdx.x * STEP_THREADS + threadIdx.x;
    const int chunk = gt / CHUNK;
    if (chunk >= nchunks) return;
    const int2 ch = chunks[chunk];
    const uint32_t cw = (uint32_t)ch.y;
    const int lane = gt % CHUNK;
    if (!((cw >> (CHUNK_LANES_SHIFT + lane)) & 1u)) return;
    const int x = (int)(cw & CHUNK_X0_MASK) + lane;
    int nb[9];
    load_row(row_nb, ch.x, nb);
    const int slot = nb[4] + x;
    T *p = static_cast<T *>(f);
    const uint32_t links = mask[slot] & LINK_MASK;
#pragma unroll
    for (int i = 0; i < 27; ++i)
        if (links & (1u << i))
            p[(int64_t)i * stride + nb[row_line<AX>(i)] + x - c_row<AX>(i)] = p[(int64_t)(26 - i) * stride + slot];
    if (periodic_row) {
        if (x == n_row - 1)
#pragma unroll
            for (int i = 0; i < 27; ++i)
                if (c_row<AX>(i) == 1) p[(int64_t)i * stride + nb[4] - 1] = p[(int64_t)i * stride + slot];
        if (x == 0)
#pragma unroll
            for (int i = 0; i < 27; ++i)
                if (c_row<AX>(i) == -1) p[(int64_t)i * stride + nb[4] + n_row] = p[(int64_t)i * stride + slot];
    }
}

// Periodic copies along the rows of the inlet/outlet nodes.
template <int P, int AX>
__global__ void __launch_bounds__(STEP_THREADS) k_fill_periodic_nodes(void *f, const int4 *bnodes, int32_t nbnodes,
                                                                      int64_t stride, int32_t n_row) {
    using T = typename Storage<P>::T;
    const int k = blockIdx.x * STEP_THREADS + threadIdx.x;
    if (k >= nbnodes) return;
    const int4 node = bnodes[(size_t)NODE_INT4S * k];
    const int x = node.z, slot = node.x, base = slot - x;
    T *p = static_cast<T *>(f);
    if (x == n_row - 1)
#pragma unroll
        for (int i = 0; i < 27; ++i)
            if (c_row<AX>(i) == 1) p[(int64_t)i * stride + base - 1] = p[(int64_t)i * stride + slot];
    if (x == 0)
#pragma unroll
        for (int i = 0; i < 27; ++i)
            if (c_row<AX>(i) == -1) p[(int64_t)i * stride + base + n_row] = p[(int64_t)i * stride + slot];
}

// Moments of the active cells k0 .. k1 - 1.  Neighbouring slots of a row along z are far
// apart in the active order, but the rows around them are written at about
// the same time, so L2 merges the 8-byte stores into whole sectors; reading
// along the active order instead took every population's sector eight times
// over (1.26 ms on the Re 3500 nozzle, now 0.5 ms).
template <int P>
__global__ void k_moments(const void *f, const int32_t *act, int64_t k0, int64_t k1, int64_t stride, float inv_scale,
                          double *rho_out, double *u_out) {
    const int64_t slot = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (slot >= stride) return;
    const int64_t k = __ldg(act + slot);
    if (k < k0 || k >= k1) return;
    double d[27], rho, ux, uy, uz;
    load_stored<P>(f, stride, (int)slot, d);
    moments_of<P>(d, inv_scale, rho, ux, uy, uz);
    if (rho_out) rho_out[k] = rho;
    if (u_out) {
        u_out[3 * k] = ux;
        u_out[3 * k + 1] = uy;
        u_out[3 * k + 2] = uz;
    }
}

__device__ __forceinline__ double wd(int i) {
    return w1<double>(cx_of(i)) * w1<double>(cy_of(i)) * w1<double>(cz_of(i));
}

template <int P>
__global__ void k_get_populations(const void *f, const int32_t *act, int64_t stride, float inv_scale,
                                  double *out27) {
    const int64_t slot = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (slot >= stride) return;
    const int64_t k = __ldg(act + slot);
    if (k < 0) return;
    double d[27];
    load_cell<P>(f, stride, (int)slot, inv_scale, d);
#pragma unroll
    for (int i = 0; i < 27; ++i) out27[27 * k + i] = wd(i) + d[i];
}

template <int P>
__device__ __forceinline__ void store_cell(void *f, int64_t stride, int slot, float scale, const double (&d)[27]) {
    using S = Storage<P>;
    typename S::T *p = static_cast<typename S::T *>(f);
#pragma unroll
    for (int i = 0; i < 27; ++i) {
        if constexpr (P == 2)
            p[(int64_t)i * stride + slot] = __float2half_rn((float)(d[i] * (double)scale));
        else
            p[(int64_t)i * stride + slot] = (typename S::T)d[i];
    }
}

template <int P>
__global__ void k_set_populations(void *f, const int32_t *act, int64_t stride, float scale, const double *in27) {
    const int64_t slot = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (slot >= stride) return;
    const int64_t k = __ldg(act + slot);
    if (k < 0) return;
    double d[27];
#pragma unroll
    for (int i = 0; i < 27; ++i) d[i] = in27[27 * k + i] - wd(i);
    store_cell<P>(f, stride, (int)slot, scale, d);
}

// Equilibrium deviations f^eq_i(rho, u) - w_i of a cell in FP64 (about 120
// operations; bound by the FP64 pipe).
__device__ __forceinline__ void eq_populations(double rho, double ux, double uy, double uz, double (&d)[27]) {
    EqLines<double> eq(rho, rho - 1.0, ux, uy, uz);
#pragma unroll
    for (int z = 0; z < 3; ++z) {
        eq.plane(z);
#pragma unroll
        for (int y = 0; y < 3; ++y) eq.line(y, d[9 * z + 3 * y], d[9 * z + 3 * y + 1], d[9 * z + 3 * y + 2]);
    }
}

// Equilibrium of the active cells k0 .. k1 - 1.
template <int P>
__global__ void k_init_eq(void *f, const int32_t *act, int64_t k0, int64_t k1, int64_t stride, float scale,
                          const double *rho, const double *u, double rho0, double ux0, double uy0, double uz0) {
    const int64_t slot = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (slot >= stride) return;
    const int64_t k = __ldg(act + slot);
    if (k < k0 || k >= k1) return;
    const double r = rho ? rho[k] : rho0;
    const double ux = u ? u[3 * k] : ux0, uy = u ? u[3 * k + 1] : uy0, uz = u ? u[3 * k + 2] : uz0;
    double d[27];
    eq_populations(r, ux, uy, uz, d);
    store_cell<P>(f, stride, (int)slot, scale, d);
}

// --------------------------------------------------------------- launchers

inline int step_blocks(int32_t nchunks) {
    const int64_t threads = (int64_t)nchunks * CHUNK;
    return (int)((threads + STEP_THREADS - 1) / STEP_THREADS);
}

// Partial-sum slots written by the fluid kernel of one step.
template <int P>
int step_fluid_blocks(int32_t nchunks) {
    return step_blocks(nchunks);
}

template <int P>
int step_stage_blocks(int device) {
    if constexpr (P == 2) {
        int per_sm = 0, sms = 0;
        cudaError_t e = cudaFuncSetAttribute(k_step_units<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, STAGE_SMEM);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_step_units<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, STAGE_SMEM);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_step_units<2>, STEP_THREADS, STAGE_SMEM);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
        if (e == cudaSuccess) return per_sm * sms;
        cudaGetLastError();
    }
    return 0;
}

template <int P>
const void *run_kernel(int mode, int row_axis) {
    if constexpr (P == 0)
        return nullptr;
    else if (mode == RATE_ONE)
        return row_axis == 2 ? (const void *)k_run<P, RATE_ONE, 2> : (const void *)k_run<P, RATE_ONE, 0>;
    else if (mode == RATE_BGK)
        return row_axis == 2 ? (const void *)k_run<P, RATE_BGK, 2> : (const void *)k_run<P, RATE_BGK, 0>;
    else
        return row_axis == 2 ? (const void *)k_run<P, RATE_GENERAL, 2> : (const void *)k_run<P, RATE_GENERAL, 0>;
}

template <int P>
int step_run_blocks(int mode, int row_axis, int device) {
    const void *fn = run_kernel<P>(mode, row_axis);
    int per_sm = 0, sms = 0, coop = 0;
    if (!fn) return 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, STEP_THREADS, 0);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, device);
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess && coop ? per_sm * sms : 0;
}

template <int P>
cudaError_t launch_run(const StepArgs &a, const RunArgs &run, int mode, int blocks, cudaStream_t s) {
    StepArgs args = a;
    RunArgs r = run;
    void *params[2] = {&args, &r};
    return cudaLaunchCooperativeKernel(run_kernel<P>(mode, a.row_axis), dim3((unsigned)blocks), dim3(STEP_THREADS), params,
                                       0, s);
}

template <int P>
int step_prefetch_ahead(int mode, bool wide, int device) {
    int per_sm = 0, sms = 0;
    cudaError_t e;
    if (mode == RATE_ONE)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &per_sm, wide ? k_step<P, RATE_ONE, true, 0> : k_step<P, RATE_ONE, false, 0>, STEP_THREADS, 0);
    else
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &per_sm, wide ? k_step<P, RATE_GENERAL, true, 0> : k_step<P, RATE_GENERAL, false, 0>, STEP_THREADS, 0);
    if (e != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    const int pct = P == 2 ? LBM_PREFETCH_AHEAD_PCT_FP16S : LBM_PREFETCH_AHEAD_PCT;
    return (int)((int64_t)per_sm * sms * pct / 100);
}

// The wall-cell and inlet/outlet kernels of a step (those not fused into
// the fluid kernel), on stream sn.
template <int P, int G, bool WD, int AX>
void launch_node_kernels(const StepArgs &a, cudaStream_t sn, bool boundary, int &launches) {
    if (a.nwnodes > 0) {  // cells with interpolated walls
        k_wall<P, G, WD, AX><<<(a.nwnodes + STEP_THREADS - 1) / STEP_THREADS, STEP_THREADS, 0, sn>>>(a);
        ++launches;
    }
    if (boundary && a.nbnodes > 0) {
        k_boundary<P, G, WD, AX><<<(a.nbnodes + STEP_THREADS - 1) / STEP_THREADS, STEP_THREADS, 0, sn>>>(a);
        ++launches;
    }
}

// One step: the node kernels go first, on the side stream when there is one
// (forked from s and joined back into it at the end), so that their few
// long-latency blocks run beside the fluid kernel instead of after it.  All
// kernels of a step read the input buffer only and write disjoint output
// elements and partial sums, so their order does not change any result.
template <int P, int G, bool WD, int AX>
cudaError_t launch_step_ax(const StepArgs &a, cudaStream_t s, const SideStream *side, int &launches) {
    const int bb = (int)((a.nbnodes + STEP_THREADS - 1) / STEP_THREADS);
    const bool tiled = G == RATE_ONE && !WD && P != 0 && a.tiles != nullptr;
    bool fluid_done = false;
    const bool fused = !tiled && LBM_FUSE_BOUNDARY && P == 1 && a.nchunks > 0;  // nodes in trailing blocks of k_step
    const bool nodes = a.nwnodes > 0 || (bb > 0 && !fused);
    const bool aside = nodes && side && side->stream;
    cudaStream_t sn = s;
    if (aside) {
        cudaError_t e = cudaEventRecord(side->fork, s);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(side->stream, side->fork, 0);
        if (e != cudaSuccess) return e;
        sn = side->stream;
    }
    launch_node_kernels<P, G, WD, AX>(a, sn, !fused, launches);
    if constexpr (G == RATE_ONE && !WD && P != 0) {
        if (tiled) {
            if constexpr (P == 2) {
                if (a.items) {  // FP16S split: pairs of fast tiles, two cells per thread; the other chunks
                    if (a.nchunks > 0) {
                        k_step<P, G, WD, AX><<<step_blocks(a.nchunks), STEP_THREADS, 0, s>>>(a);
                        ++launches;
                    }
                    if (a.nitems > 0) {
                        StepArgs b = a;  // partial sums after the chunk kernel's
                        b.partials = a.partials + (size_t)step_blocks(a.nchunks) * REDUCE_SLOTS;
                        k_step_pairs<AX><<<tile_blocks(a.nitems), STEP_THREADS, 0, s>>>(b);
                        ++launches;
                    }
                } else if (a.ntiles > 0) {
                    k_step_tiles<P, AX><<<tile_blocks(a.ntiles), STEP_THREADS, 0, s>>>(a);
                    ++launches;
                }
            } else if (a.ntiles > 0) {
                k_step_tiles<P, AX><<<tile_blocks(a.ntiles), STEP_THREADS, 0, s>>>(a);
                ++launches;
            }
        }
    }
    if constexpr (P == 2 && G == RATE_ONE && !WD) {
        if (a.units && !(a.flags & (STEP_REDUCE | STEP_STATS_FULL))) {
            const int blocks = std::min(a.stage_blocks, (a.nunits + STAGE_WARPS - 1) / STAGE_WARPS);
            k_step_units<AX><<<blocks, STEP_THREADS, STAGE_SMEM, s>>>(a);
            ++launches;
            fluid_done = true;
        }
    }
    if (!tiled && !fluid_done && a.nchunks > 0) {
        k_step<P, G, WD, AX><<<step_blocks(a.nchunks) + (fused ? bb : 0), STEP_THREADS, 0, s>>>(a);
        ++launches;
    }
    if (aside) {
        cudaError_t e = cudaEventRecord(side->join, sn);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(s, side->join, 0);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <int P, int G, bool WD>
cudaError_t launch_step_rows(const StepArgs &a, cudaStream_t s, const SideStream *side, int &launches) {
    return a.row_axis == 2 ? launch_step_ax<P, G, WD, 2>(a, s, side, launches)
                           : launch_step_ax<P, G, WD, 0>(a, s, side, launches);
}

// One time step of a lattice; launches (if not NULL) is increased by the
// number of kernels launched; side (if not NULL) is the stream of the
// wall-cell and inlet/outlet kernels.
template <int P>
cudaError_t launch_step(const StepArgs &a, int mode, cudaStream_t s, int *launches, const SideStream *side) {
    const bool wide = a.wide_offsets || a.stride > MAX_SLOTS_32;
    int n = 0;
    cudaError_t e;
    if (mode == RATE_ONE)
        e = wide ? launch_step_rows<P, RATE_ONE, true>(a, s, side, n) : launch_step_rows<P, RATE_ONE, false>(a, s, side, n);
    else if (mode == RATE_BGK && !wide)
        e = launch_step_rows<P, RATE_BGK, false>(a, s, side, n);
    else  // 64-bit offsets at omega run the general collision
        e = wide ? launch_step_rows<P, RATE_GENERAL, true>(a, s, side, n)
                 : launch_step_rows<P, RATE_GENERAL, false>(a, s, side, n);
    if (launches) *launches += n;
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <int P>
cudaError_t launch_reduce(const void *f, const int32_t *act, int64_t stride, float inv_scale, double *partials,
                          cudaStream_t s) {
    k_reduce<P><<<reduce_blocks(stride), STEP_THREADS, 0, s>>>(f, act, stride, inv_scale, partials);
    return cudaGetLastError();
}

template <int P, int AX>
void launch_fill_ghosts_ax(void *f, const uint32_t *mask, const int2 *chunks, const int4 *row_nb, int32_t nchunks,
                           const int4 *bnodes, int32_t nbnodes, int64_t stride, int32_t n_row, int32_t periodic_row,
                           cudaStream_t s) {
    const int blocks = step_blocks(nchunks);
    if (blocks > 0)
        k_fill_ghosts<P, AX><<<blocks, STEP_THREADS, 0, s>>>(f, mask, chunks, row_nb, nchunks, stride, n_row,
                                                             periodic_row);
    if (periodic_row && nbnodes > 0)
        k_fill_periodic_nodes<P, AX><<<(nbnodes + STEP_THREADS - 1) / STEP_THREADS, STEP_THREADS, 0, s>>>(
            f, bnodes, nbnodes, stride, n_row);
}

template <int P>
cudaError_t launch_fill_ghosts(void *f, const uint32_t *mask, const int2 *chunks, const int4 *row_nb,
                               int32_t nchunks, const int4 *bnodes, int32_t nbnodes, int64_t stride, int32_t n_row,
                               int32_t periodic_row, int32_t row_axis, cudaStream_t s) {
    if (row_axis == 2)
        launch_fill_ghosts_ax<P, 2>(f, mask, chunks, row_nb, nchunks, bnodes, nbnodes, stride, n_row, periodic_row, s);
    else
        launch_fill_ghosts_ax<P, 0>(f, mask, chunks, row_nb, nchunks, bnodes, nbnodes, stride, n_row, periodic_row, s);
    return cudaGetLastError();
}

inline unsigned grid_for(int64_t n, int threads) { return (unsigned)((n + threads - 1) / threads); }

template <int P>
cudaError_t launch_moments(const void *f, const int32_t *act, int64_t k0, int64_t k1, int64_t stride, float inv_scale,
                           double *rho, double *u, cudaStream_t s) {
    k_moments<P><<<grid_for(stride, 256), 256, 0, s>>>(f, act, k0, k1, stride, inv_scale, rho, u);
    return cudaGetLastError();
}

template <int P>
cudaError_t launch_get_populations(const void *f, const int32_t *act, int64_t stride, float inv_scale, double *out27,
                                   cudaStream_t s) {
    k_get_populations<P><<<grid_for(stride, 128), 128, 0, s>>>(f, act, stride, inv_scale, out27);
    return cudaGetLastError();
}

template <int P>
cudaError_t launch_set_populations(void *f, const int32_t *act, int64_t stride, float scale, const double *in27,
                                   cudaStream_t s) {
    k_set_populations<P><<<grid_for(stride, 128), 128, 0, s>>>(f, act, stride, scale, in27);
    return cudaGetLastError();
}

template <int P>
cudaError_t launch_init_eq(void *f, const int32_t *act, int64_t k0, int64_t k1, int64_t stride, float scale,
                           const double *rho, const double *u, double rho0, double ux, double uy, double uz,
                           cudaStream_t s) {
    k_init_eq<P><<<grid_for(stride, 128), 128, 0, s>>>(f, act, k0, k1, stride, scale, rho, u, rho0, ux, uy, uz);
    return cudaGetLastError();
}

#define LBM_INSTANTIATE(P)                                                                                         \
    template cudaError_t launch_step<P>(const StepArgs &, int, cudaStream_t, int *, const SideStream *);                                     \
    template int step_fluid_blocks<P>(int32_t);                                                                     \
    template int step_run_blocks<P>(int, int, int);                                                                \
    template cudaError_t launch_run<P>(const StepArgs &, const RunArgs &, int, int, cudaStream_t);                 \
    template int step_stage_blocks<P>(int);                                                                         \
    template int step_prefetch_ahead<P>(int, bool, int);                                                          \
    template cudaError_t launch_reduce<P>(const void *, const int32_t *, int64_t, float, double *, cudaStream_t);  \
    template cudaError_t launch_fill_ghosts<P>(void *, const uint32_t *, const int2 *, const int4 *, int32_t,      \
                                               const int4 *, int32_t, int64_t, int32_t, int32_t, int32_t,          \
                                               cudaStream_t);                                                      \
    template cudaError_t launch_moments<P>(const void *, const int32_t *, int64_t, int64_t, int64_t, float,         \
                                           double *, double *, cudaStream_t);                                                          \
    template cudaError_t launch_get_populations<P>(const void *, const int32_t *, int64_t, float, double *,        \
                                                   cudaStream_t);                                                  \
    template cudaError_t launch_set_populations<P>(void *, const int32_t *, int64_t, float, const double *,        \
                                                   cudaStream_t);                                                  \
    template cudaError_t launch_init_eq<P>(void *, const int32_t *, int64_t, int64_t, int64_t, float,              \
                                           const double *, const double *, double, double, double, double, cudaStream_t);

}  // namespace lbm
