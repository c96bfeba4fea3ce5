// lbm_core.cuh -- the arithmetic of one node update, written once for one
// node (float, double) and for two x-neighbours at a time (float2: the packed
// FP32 instructions apply the same operation to both nodes).
//
// The step's formulas (lbm_device.cuh) rearranged for the fewest operations:
//   * the pulled values enter as sums and differences of opposite directions;
//   * the collision's even part is E0 + c c : Q with one 2 x 2 form Q that
//     gathers the u u, u F and S terms, and E0 = 3 eps p/tau - tr Q/3 because
//     every trace term of the equilibrium and the force carries the same
//     factor 1/3 (c_s^2 = 1/3); the odd part is c . D with one vector D;
//   * the shear rate never stands alone in an interior node: S is linear in
//     (Pi, u u, u F), so its coefficients fold into those of Q;
//   * likewise the thermal odd part is c . V, its even part B0 + Kc (c.u)^2;
//   * 1/a and b/(a - b |u|^2) of the gradient solve share one reciprocal.
// FP32: 163 operations a node plus two square roots and two reciprocals; the
// direction-by-direction form took 215 (FP64 instructions of the whole step,
// square roots and reciprocals included: see k_step in lbm_kernels.cu).
//
// Every operation is spelled out (add, multiply, fused multiply-add) and no
// product feeds an addition: the compiler then has nothing to contract, so
// the scalar and the packed form, inlined into any kernel, give the same bits.
#pragma once

#include <cuda_runtime.h>

#include "lbm_device.cuh"

namespace lbm {

// ---------------------------------------------------------------- lane ops
// PTX with round-to-nearest; FP32 flushes to zero (this build's -ftz=true).
template <class L> struct LaneReal { using type = L; };
template <> struct LaneReal<float2> { using type = float; };

template <class L> __device__ __forceinline__ L lset(typename LaneReal<L>::type c) { return c; }
template <> __device__ __forceinline__ float2 lset<float2>(float c) { return make_float2(c, c); }

__device__ __forceinline__ unsigned long long lbits(float2 a) { return *reinterpret_cast<unsigned long long*>(&a); }
__device__ __forceinline__ float2 lfrom(unsigned long long u) { return *reinterpret_cast<float2*>(&u); }
__device__ __forceinline__ float ladd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double ladd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float2 ladd(float2 a, float2 b) {
    unsigned long long r;
    asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(lbits(a)), "l"(lbits(b)));
    return lfrom(r);
}
__device__ __forceinline__ float lsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double lsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float2 lsub(float2 a, float2 b) {
    unsigned long long r;
    asm("sub.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(lbits(a)), "l"(lbits(b)));
    return lfrom(r);
}
__device__ __forceinline__ float lmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double lmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float2 lmul(float2 a, float2 b) {
    unsigned long long r;
    asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(r) : "l"(lbits(a)), "l"(lbits(b)));
    return lfrom(r);
}
// a * b + c, one rounding
__device__ __forceinline__ float lfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double lfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float2 lfma(float2 a, float2 b, float2 c) {
    unsigned long long r;
    asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(lbits(a)), "l"(lbits(b)), "l"(lbits(c)));
    return lfrom(r);
}
__device__ __forceinline__ float lneg(float a) { return -a; }
__device__ __forceinline__ double lneg(double a) { return -a; }
__device__ __forceinline__ float2 lneg(float2 a) { return make_float2(-a.x, -a.y); }
// FP32: the approximate instructions (one unit in the last place)
__device__ __forceinline__ float lsqrt(float a) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}
__device__ __forceinline__ float lrcp(float a) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}
// FP64: from the hardware's approximations (about 2^-20 off) by Newton's
// iteration, once for the value and once more for its last place, so that the
// rounding of the last operation is all that is left: r' = r + r (1 - a r) twice
// for 1/a; with y ~ 1/sqrt(a), g = a y and h = y/2, d = 1/2 - g h once for both
// (g + g d ~ sqrt(a), h + h d ~ 1/(2 sqrt(a))), then g + h (a - g^2).
// Reciprocals here are of positive normal values.  Both are within 0.501 units in
// the last place, as the language's are, over 2^-900 .. 2^900.  700 x 517 with 50
// steps: 6.81 ms, about 7.1 with the language's; one iteration of third order instead
// of the two takes four FP64 instructions a node less (6.69 ms) and leaves 0.76
// and 0.51 units.
__device__ __forceinline__ double lrcp(double a) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(a));
    r = __fma_rn(r, __fma_rn(-a, r, 1.0), r);
    return __fma_rn(r, __fma_rn(-a, r, 1.0), r);
}
__device__ __forceinline__ double lsqrt(double a) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
    // The approximation takes subnormal arguments for 0 and gives infinity: the
    // root of these is 0 here.  They are |v|^2 of |v| < 1.5e-154, which the step
    // adds (times c1, or F_e/sqrt(K)) to numbers it is far below the last place of.
    if (__double2hiint(a) < 0x00100000) y = 0.0;
    double g = __dmul_rn(a, y), h = __dmul_rn(0.5, y);
    const double d = __fma_rn(-g, h, 0.5);
    g = __fma_rn(g, d, g);
    h = __fma_rn(h, d, h);
    return __fma_rn(__fma_rn(-g, g, a), h, g);
}
__device__ __forceinline__ float2 lsqrt(float2 a) { return make_float2(lsqrt(a.x), lsqrt(a.y)); }
__device__ __forceinline__ float2 lrcp(float2 a) { return make_float2(lrcp(a.x), lrcp(a.y)); }
__device__ __forceinline__ bool lfinite(float a) { return isfinite(a); }
__device__ __forceinline__ bool lfinite(double a) { return isfinite(a); }
__device__ __forceinline__ bool lfinite(float2 a) { return isfinite(a.x) && isfinite(a.y); }

// ------------------------------------------------------------ run constants
// The packed form takes every constant as a pair of equal values, laid out so
// in the kernel's parameters: a packed instruction reads its operands as
// aligned 64-bit pairs, and a pair made from one 32-bit constant costs two
// moves at each use (ALU instructions a row of pairs of the two-step kernel:
// 104 with the moves, 70 without; 59.9 -> 58.3 us a step at 2048^2, the FP16
// step unchanged within 1 %).
struct PairConst {
    float2 inv_rho0, hq_sigma, half_Q, eay, half_ax, nnuK_q2, nnuK_0, nFK_q, e1, e1_lo, e2_ie, e3_ie, qu_ie, qF_ie, cu2_ie, cuF_ie, b_0, ug_b, kc_ie, a_ep, a_const, aS, aS2, f_ScS, f_ScS2, fA_ep, f_cu, f_cF, h_sig, h_kQ, h_pT, h_u3, h_uQ, h_g, h_W, h_Wr, inv_sigma, T0, invD, rho0, gbeta, ax, omf, omT;
    float2 half, nhalf, nthird, nquarter, one, two;  // literals
    float2 w1, w5, w0, pT, n1, n5;                   // weights (core_weights)
    Cell<float2> cell;
};

// Weights of the outputs: axis, diagonal, rest, and the rest
// direction's T p term; all times the storage scale.
template <class L>
struct CoreWeights {
    L w1, w5, w0, pT, n1, n5;  // n1, n5: -w1, -w5
};
template <class R>
__host__ __device__ __forceinline__ CoreWeights<R> core_weights(const KConst<R>& k, R scale) {
    return {scale * (R(1) / R(9)), scale * w_diag<R>(), scale * (R(4) / R(9)), scale * k.h0_pT, -(scale * (R(1) / R(9))),
            -(scale * w_diag<R>())};
}
__device__ __forceinline__ CoreWeights<float2> core_weights(const PairConst& q, float) {
    return {q.w1, q.w5, q.w0, q.pT, q.n1, q.n5};
}

// The pairs of a run's constants; scale: the storage scale of the outputs.
inline PairConst make_pair_const(const KConst<float>& k, float scale) {
    PairConst q;
    auto two = [](float v) { return make_float2(v, v); };
    q.inv_rho0 = two(k.inv_rho0);
    q.hq_sigma = two(k.hq_sigma);
    q.half_Q = two(k.half_Q);
    q.eay = two(k.eay);
    q.half_ax = two(k.half_ax);
    q.nnuK_q2 = two(k.nnuK_q2);
    q.nnuK_0 = two(k.nnuK_0);
    q.nFK_q = two(k.nFK_q);
    q.e1 = two(k.e1);
    q.e1_lo = two(k.e1_lo);
    q.e2_ie = two(k.e2_ie);
    q.e3_ie = two(k.e3_ie);
    q.qu_ie = two(k.qu_ie);
    q.qF_ie = two(k.qF_ie);
    q.cu2_ie = two(k.cu2_ie);
    q.cuF_ie = two(k.cuF_ie);
    q.b_0 = two(k.b_0);
    q.ug_b = two(k.ug_b);
    q.kc_ie = two(k.kc_ie);
    q.a_ep = two(k.a_ep);
    q.a_const = two(k.a_const);
    q.aS = two(k.aS);
    q.aS2 = two(k.aS2);
    q.f_ScS = two(k.f_ScS);
    q.f_ScS2 = two(k.f_ScS2);
    q.fA_ep = two(k.fA_ep);
    q.f_cu = two(k.f_cu);
    q.f_cF = two(k.f_cF);
    q.h_sig = two(k.h_sig);
    q.h_kQ = two(k.h_kQ);
    q.h_pT = two(k.h_pT);
    q.h_u3 = two(k.h_u3);
    q.h_uQ = two(k.h_uQ);
    q.h_g = two(k.h_g);
    q.h_W = two(k.h_W);
    q.h_Wr = two(k.h_Wr);
    q.inv_sigma = two(k.inv_sigma);
    q.T0 = two(k.T0);
    q.invD = two(k.invD);
    q.rho0 = two(k.rho0);
    q.gbeta = two(k.gbeta);
    q.ax = two(k.ax);
    q.omf = two(k.omf);
    q.omT = two(k.omT);
    q.half = two(0.5f);
    q.nhalf = two(-0.5f);
    q.nthird = two(-1.0f / 3.0f);
    q.nquarter = two(-0.25f);
    q.one = two(1.0f);
    q.two = two(2.0f);
    const CoreWeights<float> w = core_weights(k, scale);
    q.w1 = two(w.w1);
    q.w5 = two(w.w5);
    q.w0 = two(w.w0);
    q.pT = two(w.pT);
    q.n1 = two(w.n1);
    q.n5 = two(w.n5);
    q.cell.eps = two(k.cell.eps);
    q.cell.ie = two(k.cell.ie);
    q.cell.elo = two(k.cell.elo);
    q.cell.eg = two(k.cell.eg);
    q.cell.eax = two(k.cell.eax);
    q.cell.heax = two(k.cell.heax);
    q.cell.c0 = two(k.cell.c0);
    q.cell.c0sq = two(k.cell.c0sq);
    q.cell.c1 = two(k.cell.c1);
    q.cell.nnuK = two(k.cell.nnuK);
    q.cell.nFK = two(k.cell.nFK);
    q.cell.e2 = two(k.cell.e2);
    q.cell.e3 = two(k.cell.e3);
    q.cell.e3_lo = two(k.cell.e3_lo);
    q.cell.re = two(k.cell.re);
    q.cell.qu = two(k.cell.qu);
    q.cell.qF = two(k.cell.qF);
    q.cell.cu2 = two(k.cell.cu2);
    q.cell.cuF = two(k.cell.cuF);
    q.cell.b = two(k.cell.b);
    q.cell.nb = two(k.cell.nb);
    q.cell.ug = two(k.cell.ug);
    q.cell.kc = two(k.cell.kc);
    return q;
}

template <class R> __device__ __forceinline__ R q_half(const KConst<R>&) { return R(0.5); }
template <class R> __device__ __forceinline__ R q_nhalf(const KConst<R>&) { return R(-0.5); }
template <class R> __device__ __forceinline__ R q_nthird(const KConst<R>&) { return R(-1) / R(3); }
template <class R> __device__ __forceinline__ R q_nquarter(const KConst<R>&) { return R(-0.25); }
template <class R> __device__ __forceinline__ R q_one(const KConst<R>&) { return R(1); }
template <class R> __device__ __forceinline__ R q_two(const KConst<R>&) { return R(2); }
__device__ __forceinline__ float2 q_half(const PairConst& q) { return q.half; }
__device__ __forceinline__ float2 q_nhalf(const PairConst& q) { return q.nhalf; }
__device__ __forceinline__ float2 q_nthird(const PairConst& q) { return q.nthird; }
__device__ __forceinline__ float2 q_nquarter(const PairConst& q) { return q.nquarter; }
__device__ __forceinline__ float2 q_one(const PairConst& q) { return q.one; }
__device__ __forceinline__ float2 q_two(const PairConst& q) { return q.two; }

// Constants at porosity e of a porosity field.  With r = (1 - e)/e the
// Kozeny-Carman and Ergun relations (Sec. 2) collapse to eps nu/K = a r^2 and
// eps F_eps/sqrt(K) = b r/e: one reciprocal, no square root.
template <class L, class Q>
__device__ __forceinline__ Cell<L> field_cell(const Q& q, L e) {
    using R = typename LaneReal<L>::type;
    Cell<L> c;
    const L ie = lrcp(e);
    const L r = lmul(lsub(q_one(q), e), ie);
    c.eps = e;
    c.ie = ie;
    c.elo = lmul(e, lfma(lneg(e), ie, q_one(q)));
    c.eg = lmul(e, q.gbeta);
    c.eax = lmul(e, q.ax);
    c.heax = lmul(e, q.half_ax);
    c.nnuK = lfma(lmul(r, r), q.nnuK_q2, q.nnuK_0);
    c.nFK = lmul(lmul(r, ie), q.nFK_q);
    c.c0 = lfma(q_nquarter(q), c.nnuK, q_half(q));
    c.c0sq = lmul(c.c0, c.c0);
    c.c1 = lmul(q_nhalf(q), c.nFK);
    c.e2 = lmul(ie, q.e2_ie);
    c.e3 = lmul(ie, q.e3_ie);
    c.e3_lo = lfma(ie, q.e3_ie, lneg(c.e3));
    c.re = lmul(ie, q.rho0);
    c.qu = lmul(ie, q.qu_ie);
    c.qF = lmul(ie, q.qF_ie);
    c.cu2 = lmul(ie, q.cu2_ie);
    c.cuF = lmul(ie, q.cuF_ie);
    c.b = lfma(q_half(q), ie, q.b_0);
    c.nb = lfma(q_nhalf(q), ie, lneg(q.b_0));
    c.ug = lmul(c.b, q.ug_b);
    c.kc = lmul(ie, q.kc_ie);
    return c;
}

// Constants of node (x, y).
template <class R>
__device__ __forceinline__ Cell<R> node_cell(const KConst<R>& k, int x, int y) {
    return k.eps_field ? field_cell<R>(k, k.eps_field[(long long)y * k.nx + x]) : k.cell;
}

// eps a_y of a node in row y: uniform porosity without a profile has it as a
// constant.
template <class L, class R, class Q>
__device__ __forceinline__ L eps_ay(const KConst<R>& k, const Q& q, const Cell<L>& c, int y) {
    return k.ay_row || k.eps_field ? lmul(c.eps, lset<L>(row_ay(k, y))) : q.eay;
}

// ------------------------------------------------------------------ moments

// What the collision needs of a node's moments (Secs. 3.1-3.3); ep = eps p,
// Px = Pi_xx - eps p, Py likewise.
template <class L>
struct CoreState {
    L th, T, ux, uy, Fx, Fy, ep, Px, Py, Pxy, gx, gy;
};

// Sum of the pulled thermal deviations, in the order core_moments adds them.
template <class L>
__device__ __forceinline__ L core_hsum(const L* h) {
    return ladd(ladd(ladd(ladd(h[1], h[3]), ladd(h[2], h[4])), ladd(ladd(h[5], h[7]), ladd(h[6], h[8]))), h[0]);
}
// What the last two additions of core_hsum rounded off (exact: Knuth's two-sum).
template <class L>
__device__ __forceinline__ L core_hsum_rest(const L* h) {
    auto rest = [](L a, L b) {
        const L s = ladd(a, b), v = lsub(s, a);
        return ladd(lsub(a, lsub(s, v)), lsub(b, v));
    };
    const L A = ladd(ladd(h[1], h[3]), ladd(h[2], h[4])), B = ladd(ladd(h[5], h[7]), ladd(h[6], h[8]));
    return ladd(rest(A, B), rest(ladd(A, B), h[0]));
}
// T - T0 from that sum: (sum + Q/2)/sigma.
template <class L, class Q>
__device__ __forceinline__ L core_theta(const Q& q, L hsum) {
    return lfma(hsum, q.inv_sigma, q.hq_sigma);
}

template <class L, class Q>
__device__ __forceinline__ CoreState<L> core_moments(const Q& q, const Cell<L>& c, L eay, const L* f,
                                                     const L* h) {
    using R = typename LaneReal<L>::type;
    CoreState<L> s;
    const L half = q_half(q);
    s.th = core_theta(q, core_hsum(h));
    s.T = ladd(q.T0, s.th);
    const L s13 = ladd(f[1], f[3]), s24 = ladd(f[2], f[4]), s57 = ladd(f[5], f[7]), s68 = ladd(f[6], f[8]);
    const L d57 = lsub(f[5], f[7]), d86 = lsub(f[8], f[6]);
    const L mx = ladd(lsub(f[1], f[3]), ladd(d57, d86));
    const L my = ladd(lsub(f[2], f[4]), lsub(d57, d86));
    const L d58 = ladd(s57, s68);
    const L Pyy = ladd(s24, d58);
    const L Pxx = ladd(s13, d58);
    const L sf = ladd(s13, Pyy);
    s.Pxy = lsub(s57, s68);
    const L eGy = lfma(c.eg, s.th, eay);  // eps G_y
    const L ir = q.inv_rho0;
    const L vx = lfma(mx, ir, c.heax);
    const L vy = lfma(my, ir, lmul(half, eGy));
    const L vmag = lsqrt(lfma(vx, vx, lmul(vy, vy)));
    const L iden = lrcp(ladd(c.c0, lsqrt(lfma(c.c1, vmag, c.c0sq))));
    const L um = lmul(vmag, iden);  // |u| = |v| / (c0 + sqrt(c0^2 + c1 |v|)): no further square root
    s.ux = lmul(vx, iden);
    s.uy = lmul(vy, iden);
    const L uu = lfma(s.ux, s.ux, lmul(s.uy, s.uy));
    const L nd = lfma(c.nFK, um, c.nnuK);
    s.Fx = lfma(nd, s.ux, c.eax);
    s.Fy = lfma(nd, s.uy, eGy);
    const L uF = lfma(s.ux, s.Fx, lmul(s.uy, s.Fy));
    L ep = lfma(c.e2, uF, lmul(c.e3, uu));
    if constexpr (sizeof(R) == 4) ep = lfma(q.e1_lo, sf, lfma(c.e3_lo, uu, ep));
    s.ep = lfma(q.e1, sf, ep);
    s.Px = lsub(Pxx, s.ep);
    s.Py = lsub(Pyy, s.ep);
    // grad T: (a I - b u u^T) grad T = N
    const L h57 = lsub(h[5], h[7]), h86 = lsub(h[8], h[6]);
    const L hx = ladd(lsub(h[1], h[3]), ladd(h57, h86));
    const L hy = ladd(lsub(h[2], h[4]), lsub(h57, h86));
    const L qT = lsub(q.hq_sigma, s.T), Th = lmul(half, s.T);
    const L Nx = lfma(s.ux, qT, lfma(Th, s.Fx, hx));
    const L Ny = lfma(s.uy, qT, lfma(Th, s.Fy, hy));
    const L a = lfma(q.a_ep, s.ep, q.a_const);
    const L d = lfma(c.nb, uu, a);
    const L r = lrcp(lmul(a, d));  // 1/a = d r, 1/d = a r
    const L ia = lmul(d, r);
    const L t = lmul(lmul(c.b, lfma(s.ux, Nx, lmul(s.uy, Ny))), r);
    s.gx = lfma(t, s.ux, lmul(ia, Nx));
    s.gy = lfma(t, s.uy, lmul(ia, Ny));
    return s;
}

// Shear rate from the state (walls and the moment state store it).
template <class L>
struct Shear {
    L xx, yy, xy;
};
template <class L, class Q>
__device__ __forceinline__ Shear<L> core_shear(const Q& q, const Cell<L>& c, const CoreState<L>& s) {
    const L D = q.invD;
    const L dx = lsub(s.Fx, s.ux), dy = lsub(s.Fy, s.uy);
    const L rx = lmul(c.re, s.ux), ry = lmul(c.re, s.uy);
    Shear<L> S;
    S.xx = lmul(D, lfma(rx, dx, s.Px));
    S.yy = lmul(D, lfma(ry, dy, s.Py));
    S.xy = lmul(D, lfma(q_half(q), lfma(rx, dy, lmul(ry, dx)), s.Pxy));
    return S;
}

// The form Q of the even flow part (Q2 = 2 Q_xy): from the pulled second
// moments (interior nodes) ...
template <class L, class Q>
__device__ __forceinline__ void core_form(const Q& q, const Cell<L>& c, const CoreState<L>& s, L& Qxx, L& Qyy,
                                          L& Q2) {
    const L al = q.aS;
    const L tx = lfma(c.qu, s.ux, lmul(c.qF, s.Fx)), ty = lfma(c.qu, s.uy, lmul(c.qF, s.Fy));
    Qxx = lfma(s.ux, tx, lmul(al, s.Px));
    Qyy = lfma(s.uy, ty, lmul(al, s.Py));
    Q2 = lfma(s.ux, ty, lfma(s.uy, tx, lmul(q.aS2, s.Pxy)));
}
// ... or from an explicit shear rate (walls, moment state).
template <bool SOURCES, class L, class Q>
__device__ __forceinline__ void shear_form(const Q& q, const Cell<L>& c, L ux, L uy, L Fx, L Fy,
                                           const Shear<L>& S, L& Qxx, L& Qyy, L& Q2) {
    const L fs = q.f_ScS;
    const L tx = SOURCES ? lfma(c.cu2, ux, lmul(c.cuF, Fx)) : lmul(c.cu2, ux);
    const L ty = SOURCES ? lfma(c.cu2, uy, lmul(c.cuF, Fy)) : lmul(c.cu2, uy);
    Qxx = lfma(ux, tx, lmul(fs, S.xx));
    Qyy = lfma(uy, ty, lmul(fs, S.yy));
    Q2 = lfma(ux, ty, lfma(uy, tx, lmul(q.f_ScS2, S.xy)));
}

// Collision: f* = (1 - 1/tau) f + f^eq/tau + F_i and g* likewise, from the
// state and the form Q.  TAU1: tau_f = tau_T = 1 (f, h are not read); then
// wscale multiplies every output (the FP16 storage scale).  SOURCES = false
// keeps the equilibria alone.  REST: u = 0 (a wall without slip), whose terms
// are left out (the same values: they are products with zero).
template <bool TAU1, bool SOURCES, bool REST = false, class L, class Q>
__device__ __forceinline__ void core_emit(const Q& q, const Cell<L>& c, const CoreState<L>& s, L Qxx, L Qyy,
                                          L Q2, const L* f, const L* h, L* fo, L* ho,
                                          typename LaneReal<L>::type wscale) {
    const CoreWeights<L> w_ = core_weights(q, wscale);
    const L w1 = w_.w1;
    const L nthird = q_nthird(q);
    // out_i, out_j = w (e +- d) of two opposite directions.  The smaller of
    // the two parts is scaled by w first, so that each output is rounded once
    // at its own size: in the flow e ~ u^2 < d ~ u, in the temperature d < e.
    auto put_f = [&](int i, int j, const L& w, const L& n, const L& e, const L& d) {
        const L b = lmul(w, e);
        fo[i] = lfma(w, d, TAU1 ? b : lfma(q.omf, f[i], b));
        fo[j] = lfma(n, d, TAU1 ? b : lfma(q.omf, f[j], b));
    };
    {
        const L tr = ladd(Qxx, Qyy);
        const L E = lfma(nthird, tr, lmul(q.fA_ep, s.ep));
        const L Ed = ladd(E, tr);
        const L fu = q.f_cu, fF = q.f_cF;
        L Dx, Dy;
        if constexpr (REST) {
            Dx = lmul(fF, s.Fx);
            Dy = lmul(fF, s.Fy);
        } else {
            Dx = SOURCES ? lfma(fu, s.ux, lmul(fF, s.Fx)) : lmul(fu, s.ux);
            Dy = SOURCES ? lfma(fu, s.uy, lmul(fF, s.Fy)) : lmul(fu, s.uy);
        }
        const L w5 = w_.w5;
        put_f(1, 3, w1, w_.n1, ladd(E, Qxx), Dx);
        put_f(2, 4, w1, w_.n1, ladd(E, Qyy), Dy);
        put_f(5, 7, w5, w_.n5, ladd(Ed, Q2), SOURCES ? ladd(Dx, Dy) : lfma(fu, s.uy, Dx));
        put_f(6, 8, w5, w_.n5, lsub(Ed, Q2), SOURCES ? lsub(Dy, Dx) : lfma(lneg(q.f_cu), s.ux, Dy));
    }
    {
        // even part: sigma theta plus small terms, summed among themselves first
        const L T = s.T, Tep = lmul(T, s.ep);
        const L th = lmul(q.h_sig, s.th);
        L kx = L(), ky = L(), tr = L();
        if constexpr (!REST) {
            const L kc = lmul(c.kc, T);
            kx = lmul(kc, s.ux);
            ky = lmul(kc, s.uy);
            tr = lfma(kx, s.ux, lmul(ky, s.uy));
        }
        const L m0 = REST ? q.h_kQ : SOURCES ? lfma(nthird, tr, q.h_kQ) : lmul(nthird, tr);
        // h + (w sum h - h)/tau + w (small +- d): the difference is small, so
        // the output is rounded once at its own size here too; sigma theta =
        // sum h + Q/2, and what the sum in R misses joins the small terms
        const L itT = lsub(q_one(q), q.omT);
        L tr0, m1 = m0;
        if constexpr (!TAU1) {
            tr0 = core_hsum(h);
            m1 = lfma(itT, ladd(core_hsum_rest(h), q.half_Q), m0);
        }
        const L m = lfma(q.h_pT, Tep, m1);
        const L md = REST ? m : SOURCES ? ladd(m, tr) : lfma(q_one(q), tr, m);
        L Vx, Vy;
        if constexpr (REST) {
            const L hg = lfma(q.h_Wr, s.ep, q.h_g), hT = lmul(q.h_W, T);
            Vx = lfma(hg, s.gx, lmul(hT, s.Fx));
            Vy = lfma(hg, s.gy, lmul(hT, s.Fy));
        } else if constexpr (SOURCES) {
            const L K = lfma(q.h_u3, T, lfma(c.ug, lfma(s.ux, s.gx, lmul(s.uy, s.gy)), q.h_uQ));
            const L hg = lfma(q.h_Wr, s.ep, q.h_g), hT = lmul(q.h_W, T);
            Vx = lfma(K, s.ux, lfma(hg, s.gx, lmul(hT, s.Fx)));
            Vy = lfma(K, s.uy, lfma(hg, s.gy, lmul(hT, s.Fy)));
        } else {
            const L K = lmul(q.h_u3, T), hg = q.h_g;
            Vx = lfma(K, s.ux, lmul(hg, s.gx));
            Vy = lfma(K, s.uy, lmul(hg, s.gy));
        }
        const L w5 = w_.w5;
        auto relax = [&](const L& w, const L& small, const L& in) {
            return ladd(in, lfma(itT, lfma(w, tr0, lneg(in)), lmul(w, small)));
        };
        auto put_h = [&](int i, int j, const L& w, const L& small, const L& d) {
            if constexpr (TAU1) {
                const L e = ladd(th, small), b = lmul(w, d);
                ho[i] = lfma(w, e, b);
                ho[j] = lfma(w, e, lneg(b));
            } else {
                ho[i] = relax(w, ladd(small, d), h[i]);
                ho[j] = relax(w, lsub(small, d), h[j]);
            }
        };
        if constexpr (REST) {
            put_h(1, 3, w1, m, Vx);
            put_h(2, 4, w1, m, Vy);
            put_h(5, 7, w5, m, ladd(Vx, Vy));
            put_h(6, 8, w5, m, lsub(Vy, Vx));
        } else {
            put_h(1, 3, w1, lfma(kx, s.ux, m), Vx);
            put_h(2, 4, w1, lfma(ky, s.uy, m), Vy);
            const L k2 = lmul(q_two(q), kx);
            put_h(5, 7, w5, lfma(k2, s.uy, md), ladd(Vx, Vy));
            put_h(6, 8, w5, lfma(lneg(k2), s.uy, md), lsub(Vy, Vx));
        }
        const L w0 = w_.w0;
        const L pT = w_.pT;
        if constexpr (TAU1) ho[0] = lfma(w0, th, lfma(w0, m0, lmul(pT, Tep)));
        else ho[0] = ladd(h[0], lfma(itT, lfma(w0, tr0, lneg(h[0])), lfma(w0, m1, lmul(pT, Tep))));
    }
}

// Interior node: moments, then the collision.  (The rest direction's thermal
// value ho[0] is finite only if T and u are: the caller's watchdog looks at it.)
template <bool TAU1, class L, class Q>
__device__ __forceinline__ void core_interior(const Q& q, const Cell<L>& c, L eay, const L* f, const L* h, L* fo, L* ho,
                                              typename LaneReal<L>::type wscale = 1) {
    const CoreState<L> s = core_moments(q, c, eay, f, h);
    L Qxx, Qyy, Q2;
    core_form(q, c, s, Qxx, Qyy, Q2);
    core_emit<TAU1, true>(q, c, s, Qxx, Qyy, Q2, f, h, fo, ho, wscale);
}

// Moment state (tau_f = tau_T = 1): the nine stored moments of a state ...
template <class L, class Q>
__device__ __forceinline__ void stored_moments(const Q& q, const Cell<L>& c, const CoreState<L>& s, L* m) {
    const Shear<L> S = core_shear(q, c, s);
    m[MP] = lmul(s.ep, c.ie);
    m[MUX] = s.ux;
    m[MUY] = s.uy;
    m[MSXX] = S.xx;
    m[MSYY] = S.yy;
    m[MSXY] = S.xy;
    m[MTH] = s.th;
    m[MGX] = s.gx;
    m[MGY] = s.gy;
}
// ... and the populations of a node from them; F is recomputed from (u, T) as in
// core_moments (and, for a wall node, as in core_boundary).
template <bool SOURCES, class L, class Q>
__device__ __forceinline__ void expand_moments(const Q& q, const Cell<L>& c, L eay, const L* m, L* fo, L* ho) {
    CoreState<L> s;
    s.ux = m[MUX];
    s.uy = m[MUY];
    s.th = m[MTH];
    s.gx = m[MGX];
    s.gy = m[MGY];
    s.T = ladd(q.T0, s.th);
    const L uu = lfma(s.ux, s.ux, lmul(s.uy, s.uy));
    const L nd = lfma(c.nFK, lsqrt(uu), c.nnuK);
    s.Fx = lfma(nd, s.ux, c.eax);
    s.Fy = lfma(nd, s.uy, lfma(c.eg, s.th, eay));
    s.ep = lfma(c.eps, m[MP], lmul(c.elo, m[MP]));  // the inverse of p = ep ie as stored (e ie != 1)
    const Shear<L> S = {m[MSXX], m[MSYY], m[MSXY]};
    L Qxx, Qyy, Q2;
    shear_form<SOURCES>(q, c, s.ux, s.uy, s.Fx, s.Fy, S, Qxx, Qyy, Q2);
    core_emit<true, SOURCES>(q, c, s, Qxx, Qyy, Q2, (const L*)nullptr, (const L*)nullptr, fo, ho,
                             typename LaneReal<L>::type(1));
}

// Boundary state b of a wall node (Sec. 3.4); S(x_f) stands beside it.  At tau_f =
// tau_T = 1 the extrapolated non-equilibrium part carries the factor 1 - 1/tau =
// 0, and the node is the collision of b alone.  s: state of x_f on entry, b on
// return; cs / cb: constants of x_f and of the node, thff: T(x_ff) - T0, thb: the
// Dirichlet T_b - T0 where `given`.
template <class R>
__device__ __forceinline__ void core_boundary(const KConst<R>& k, const Cell<R>& cs, const Cell<R>& cb, R eay_b,
                                              R ubx, R uby, R ubm, bool given, bool fixgx, bool fixgy, R thb, R thff,
                                              CoreState<R>& s) {
    s.ux = ubx;
    s.uy = uby;
    if (given) {
        s.th = thb;
    } else {
        // Eq. (TNEESApGra) with zero normal gradient
        s.th = lmul(R(1) / R(3), lfma(R(4), s.th, lneg(thff)));
        if (fixgx) s.gx = R(0);
        if (fixgy) s.gy = R(0);
    }
    s.T = ladd(k.T0, s.th);
    // p(x_f) at the wall node's own porosity
    if (k.eps_field) s.ep = lmul(lmul(s.ep, cs.ie), cb.eps);
    const R nd = lfma(cb.nFK, ubm, cb.nnuK);
    s.Fx = lfma(nd, s.ux, cb.eax);
    s.Fy = lfma(nd, s.uy, lfma(cb.eg, s.th, eay_b));
}

// Wall node at any relaxation times: f* = (1 - 1/tau) [f(x_f) - f^eq(s)] +
// f^eq(b) + F_i(b) and g* likewise (Eqs. NEESVel, TNEESAp), the two equilibria and the
// sources gathered into one scalar, form and vector per distribution as in
// core_emit.  s, S: state and shear rate of x_f, b: the boundary state
// (core_boundary), cs / cb their constants, f, h: the values pulled at x_f.
template <class R>
__device__ __forceinline__ void wall_emit(const KConst<R>& k, const Cell<R>& cs, const Cell<R>& cb, const CoreState<R>& s,
                                          const Shear<R>& S, const CoreState<R>& b, const R* f, const R* h, R* fo, R* ho) {
    const CoreWeights<R> w_ = core_weights(k, R(1));
    const R third = R(1) / R(3);
    {
        const R m = -k.omf, c2 = lmul(R(4.5), cs.re), cb2 = lmul(R(4.5), cb.re), cF = lmul(lmul(R(9), k.kf), cb.re);
        const R sx = lmul(c2, s.ux), sy = lmul(c2, s.uy);
        const R tx = lfma(cb2, b.ux, lmul(cF, b.Fx)), ty = lfma(cb2, b.uy, lmul(cF, b.Fy));
        const R fS = lmul(lmul(lmul(R(1.5), k.rho0), k.A), ladd(R(1), m));  // S is that of x_f in both
        const R Qxx = lfma(m, lmul(s.ux, sx), lfma(b.ux, tx, lmul(fS, S.xx)));
        const R Qyy = lfma(m, lmul(s.uy, sy), lfma(b.uy, ty, lmul(fS, S.yy)));
        const R Q2 = lfma(m, lfma(s.ux, sy, lmul(s.uy, sx)), lfma(b.ux, ty, lfma(b.uy, tx, lmul(lmul(R(2), fS), S.xy))));
        const R tr = ladd(Qxx, Qyy), E = lfma(-third, tr, lmul(R(3), lfma(m, s.ep, b.ep))), Ed = ladd(E, tr);
        const R c1 = lmul(R(3), k.rho0), cf = lmul(c1, k.kf);
        const R Dx = lfma(c1, lfma(m, s.ux, b.ux), lmul(cf, b.Fx)), Dy = lfma(c1, lfma(m, s.uy, b.uy), lmul(cf, b.Fy));
        auto put = [&](int i, int j, R w, R n, R e, R d) {
            const R we = lmul(w, e);
            fo[i] = lfma(w, d, lfma(k.omf, f[i], we));
            fo[j] = lfma(n, d, lfma(k.omf, f[j], we));
        };
        put(1, 3, w_.w1, w_.n1, ladd(E, Qxx), Dx);
        put(2, 4, w_.w1, w_.n1, ladd(E, Qyy), Dy);
        put(5, 7, w_.w5, w_.n5, ladd(Ed, Q2), ladd(Dx, Dy));
        put(6, 8, w_.w5, w_.n5, lsub(Ed, Q2), lsub(Dy, Dx));
    }
    {
        const R m = -k.omT, ks = lmul(lmul(R(4.5), cs.ie), s.T), kb = lmul(lmul(R(4.5), cb.ie), b.T);
        const R sx = lmul(ks, s.ux), sy = lmul(ks, s.uy), tx = lmul(kb, b.ux), ty = lmul(kb, b.uy);
        const R Kxx = lfma(m, lmul(sx, s.ux), lmul(tx, b.ux)), Kyy = lfma(m, lmul(sy, s.uy), lmul(ty, b.uy));
        const R K2 = lmul(R(2), lfma(m, lmul(sx, s.uy), lmul(tx, b.uy)));
        const R tr = ladd(Kxx, Kyy), th = lmul(k.sigma, lfma(m, s.th, b.th)), m0 = lfma(-third, tr, k.h_kQ);
        const R pT = lmul(lmul(R(3), k.inv_rho0), lfma(m, lmul(s.T, s.ep), lmul(b.T, b.ep)));
        const R e = ladd(m0, pT), ed = ladd(e, tr);
        const R sB = lmul(k.sigma, k.B), hg = lfma(k.h_Wr, b.ep, sB), hT = lmul(k.h_W, b.T), T3 = lmul(R(3), s.T);
        const R K = lfma(R(3), b.T, lfma(cb.ug, lfma(b.ux, b.gx, lmul(b.uy, b.gy)), k.h_uQ));
        const R Vx = lfma(m, lfma(T3, s.ux, lmul(sB, s.gx)), lfma(K, b.ux, lfma(hg, b.gx, lmul(hT, b.Fx))));
        const R Vy = lfma(m, lfma(T3, s.uy, lmul(sB, s.gy)), lfma(K, b.uy, lfma(hg, b.gy, lmul(hT, b.Fy))));
        auto put = [&](int i, int j, R w, R small, R d) {
            const R even = ladd(th, small), wd = lmul(w, d);
            ho[i] = lfma(w, even, lfma(k.omT, h[i], wd));
            ho[j] = lfma(w, even, lfma(k.omT, h[j], lneg(wd)));
        };
        put(1, 3, w_.w1, ladd(e, Kxx), Vx);
        put(2, 4, w_.w1, ladd(e, Kyy), Vy);
        put(5, 7, w_.w5, ladd(ed, K2), ladd(Vx, Vy));
        put(6, 8, w_.w5, lsub(ed, K2), lsub(Vy, Vx));
        ho[0] = lfma(w_.w0, ladd(th, m0), lfma(k.omT, h[0], lmul(-(R(5) / R(9)), pT)));
    }
}

}  // namespace lbm
