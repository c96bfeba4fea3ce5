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
__device__ __forceinline__ double lsqrt(double a) { return sqrt(a); }
__device__ __forceinline__ double lrcp(double a) { return 1.0 / a; }
__device__ __forceinline__ float2 lsqrt(float2 a) { return make_float2(lsqrt(a.x), lsqrt(a.y)); }
__device__ __forceinline__ float2 lrcp(float2 a) { return make_float2(lrcp(a.x), lrcp(a.y)); }
__device__ __forceinline__ bool lfinite(float a) { return isfinite(a); }
__device__ __forceinline__ bool lfinite(double a) { return isfinite(a); }
__device__ __forceinline__ bool lfinite(float2 a) { return isfinite(a.x) && isfinite(a.y); }

// ------------------------------------------------------------ node constants

// The run's own constants (uniform porosity), one copy per lane.
template <class L, class R>
__device__ __forceinline__ Cell<L> uniform_cell(const KConst<R>& k) {
    Cell<L> c;
    c.eps = lset<L>(k.cell.eps);
    c.ie = lset<L>(k.cell.ie);
    c.eg = lset<L>(k.cell.eg);
    c.eax = lset<L>(k.cell.eax);
    c.heax = lset<L>(k.cell.heax);
    c.c0 = lset<L>(k.cell.c0);
    c.c0sq = lset<L>(k.cell.c0sq);
    c.c1 = lset<L>(k.cell.c1);
    c.ih = lset<L>(k.cell.ih);
    c.il = lset<L>(k.cell.il);
    c.ci = lset<L>(k.cell.ci);
    c.nnuK = lset<L>(k.cell.nnuK);
    c.nFK = lset<L>(k.cell.nFK);
    c.e2 = lset<L>(k.cell.e2);
    c.e3 = lset<L>(k.cell.e3);
    c.re = lset<L>(k.cell.re);
    c.qu = lset<L>(k.cell.qu);
    c.qF = lset<L>(k.cell.qF);
    c.cu2 = lset<L>(k.cell.cu2);
    c.cuF = lset<L>(k.cell.cuF);
    c.b = lset<L>(k.cell.b);
    c.nb = lset<L>(k.cell.nb);
    c.ug = lset<L>(k.cell.ug);
    c.kc = lset<L>(k.cell.kc);
    return c;
}

// Constants at porosity e of a porosity field.  With q = (1 - e)/e the
// Kozeny-Carman and Ergun relations (Sec. 2) collapse to eps nu/K = a q^2 and
// eps F_eps/sqrt(K) = b q/e: one reciprocal, no square root.
template <class L, class R>
__device__ __forceinline__ Cell<L> field_cell(const KConst<R>& k, L e) {
    Cell<L> c;
    const L ie = lrcp(e);
    const L q = lmul(lsub(lset<L>(R(1)), e), ie);
    c.eps = e;
    c.ie = ie;
    c.eg = lmul(e, lset<L>(k.gbeta));
    c.eax = lmul(e, lset<L>(k.ax));
    c.heax = lmul(e, lset<L>(k.half_ax));
    c.nnuK = lmul(lmul(q, q), lset<L>(k.nnuK_q2));
    c.nFK = lmul(lmul(q, ie), lset<L>(k.nFK_q));
    c.c0 = lfma(lset<L>(R(-0.25)), c.nnuK, lset<L>(R(0.5)));
    c.c0sq = lmul(c.c0, c.c0);
    c.c1 = lmul(lset<L>(R(-0.5)), c.nFK);
    const L d = lfma(lset<L>(R(-0.5)), c.nnuK, lset<L>(R(1)));  // 2 c0
    c.ih = lrcp(d);
    c.il = lmul(c.ih, lfma(lneg(d), c.ih, lset<L>(R(1))));
    if constexpr (sizeof(R) == 4) c.il = lfma(c.ih, lset<L>(k.gain), c.il);
    c.ci = lneg(lmul(c.c1, c.ih));
    c.e2 = lmul(ie, lset<L>(k.e2_ie));
    c.e3 = lmul(ie, lset<L>(k.e3_ie));
    c.re = lmul(ie, lset<L>(k.rho0));
    c.qu = lmul(ie, lset<L>(k.qu_ie));
    c.qF = lmul(ie, lset<L>(k.qF_ie));
    c.cu2 = lmul(ie, lset<L>(k.cu2_ie));
    c.cuF = lmul(ie, lset<L>(k.cuF_ie));
    c.b = lfma(lset<L>(R(0.5)), ie, lset<L>(k.b_0));
    c.nb = lfma(lset<L>(R(-0.5)), ie, lset<L>(-k.b_0));
    c.ug = lmul(c.b, lset<L>(k.ug_b));
    c.kc = lmul(ie, lset<L>(k.kc_ie));
    return c;
}

// Constants of node (x, y).
template <class R>
__device__ __forceinline__ Cell<R> node_cell(const KConst<R>& k, int x, int y) {
    return k.eps_field ? field_cell<R>(k, k.eps_field[(long long)y * k.nx + x]) : uniform_cell<R>(k);
}

// eps a_y of a node in row y: uniform porosity without a profile has it as a
// constant.
template <class L, class R>
__device__ __forceinline__ L eps_ay(const KConst<R>& k, const Cell<L>& c, int y) {
    return k.ay_row || k.eps_field ? lmul(c.eps, lset<L>(row_ay(k, y))) : lset<L>(k.eay);
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
template <class L, class R>
__device__ __forceinline__ L core_theta(const KConst<R>& k, L hsum) {
    return lfma(hsum, lset<L>(k.inv_sigma), lset<L>(k.hq_sigma));
}

template <class L, class R>
__device__ __forceinline__ CoreState<L> core_moments(const KConst<R>& k, const Cell<L>& c, L eay, const L* f,
                                                     const L* h) {
    CoreState<L> s;
    const L half = lset<L>(R(0.5));
    s.th = core_theta(k, core_hsum(h));
    s.T = ladd(lset<L>(k.T0), s.th);
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
    const L ir = lset<L>(k.inv_rho0);
    const L vx = lfma(mx, ir, c.heax);
    const L vy = lfma(my, ir, lmul(half, eGy));
    const L vmag = lsqrt(lfma(vx, vx, lmul(vy, vy)));
    const L iden = lrcp(ladd(c.c0, lsqrt(lfma(c.c1, vmag, c.c0sq))));
    const L um = lmul(vmag, iden);  // |u| = |v| / (c0 + sqrt(c0^2 + c1 |v|)): no further square root
    if constexpr (sizeof(R) == 4) {
        // The same quotient as v/(2 c0) less a small part: with
        // sqrt(c0^2 + c1 |v|) - c0 = c1 |u|, 1/den = ih - ih c1 |u|/den,
        // ih + il = 1/(2 c0).  v iden would carry the rounding of den, the same
        // at every step where c1 |v| is small: a gain or loss of momentum of up
        // to 1e-7 a step that builds up.
        const L q = lfma(lmul(c.ci, um), iden, c.il);
        s.ux = lfma(vx, c.ih, lmul(vx, q));
        s.uy = lfma(vy, c.ih, lmul(vy, q));
    } else {
        s.ux = lmul(vx, iden);
        s.uy = lmul(vy, iden);
    }
    const L uu = lfma(s.ux, s.ux, lmul(s.uy, s.uy));
    const L nd = lfma(c.nFK, um, c.nnuK);
    s.Fx = lfma(nd, s.ux, c.eax);
    s.Fy = lfma(nd, s.uy, eGy);
    const L uF = lfma(s.ux, s.Fx, lmul(s.uy, s.Fy));
    L ep = lfma(c.e2, uF, lmul(c.e3, uu));
    if constexpr (sizeof(R) == 4) ep = lfma(lset<L>(k.e1_lo), sf, ep);
    s.ep = lfma(lset<L>(k.e1), sf, ep);
    s.Px = lsub(Pxx, s.ep);
    s.Py = lsub(Pyy, s.ep);
    // grad T: (a I - b u u^T) grad T = N
    const L h57 = lsub(h[5], h[7]), h86 = lsub(h[8], h[6]);
    const L hx = ladd(lsub(h[1], h[3]), ladd(h57, h86));
    const L hy = ladd(lsub(h[2], h[4]), lsub(h57, h86));
    const L qT = lsub(lset<L>(k.hq_sigma), s.T), Th = lmul(half, s.T);
    const L Nx = lfma(s.ux, qT, lfma(Th, s.Fx, hx));
    const L Ny = lfma(s.uy, qT, lfma(Th, s.Fy, hy));
    const L a = lfma(lset<L>(k.a_ep), s.ep, lset<L>(k.a_const));
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
template <class L, class R>
__device__ __forceinline__ Shear<L> core_shear(const KConst<R>& k, const Cell<L>& c, const CoreState<L>& s) {
    const L D = lset<L>(k.invD);
    const L dx = lsub(s.Fx, s.ux), dy = lsub(s.Fy, s.uy);
    const L rx = lmul(c.re, s.ux), ry = lmul(c.re, s.uy);
    Shear<L> S;
    S.xx = lmul(D, lfma(rx, dx, s.Px));
    S.yy = lmul(D, lfma(ry, dy, s.Py));
    S.xy = lmul(D, lfma(lset<L>(R(0.5)), lfma(rx, dy, lmul(ry, dx)), s.Pxy));
    return S;
}

// The form Q of the even flow part (Q2 = 2 Q_xy): from the pulled second
// moments (interior nodes) ...
template <class L, class R>
__device__ __forceinline__ void core_form(const KConst<R>& k, const Cell<L>& c, const CoreState<L>& s, L& Qxx, L& Qyy,
                                          L& Q2) {
    const L al = lset<L>(k.aS);
    const L tx = lfma(c.qu, s.ux, lmul(c.qF, s.Fx)), ty = lfma(c.qu, s.uy, lmul(c.qF, s.Fy));
    Qxx = lfma(s.ux, tx, lmul(al, s.Px));
    Qyy = lfma(s.uy, ty, lmul(al, s.Py));
    Q2 = lfma(s.ux, ty, lfma(s.uy, tx, lmul(lset<L>(k.aS2), s.Pxy)));
}
// ... or from an explicit shear rate (walls, moment state).
template <bool SOURCES, class L, class R>
__device__ __forceinline__ void shear_form(const KConst<R>& k, const Cell<L>& c, L ux, L uy, L Fx, L Fy,
                                           const Shear<L>& S, L& Qxx, L& Qyy, L& Q2) {
    const L fs = lset<L>(k.f_ScS);
    const L tx = SOURCES ? lfma(c.cu2, ux, lmul(c.cuF, Fx)) : lmul(c.cu2, ux);
    const L ty = SOURCES ? lfma(c.cu2, uy, lmul(c.cuF, Fy)) : lmul(c.cu2, uy);
    Qxx = lfma(ux, tx, lmul(fs, S.xx));
    Qyy = lfma(uy, ty, lmul(fs, S.yy));
    Q2 = lfma(ux, ty, lfma(uy, tx, lmul(lset<L>(k.f_ScS2), S.xy)));
}

// Collision: f* = (1 - 1/tau) f + f^eq/tau + F_i and g* likewise, from the
// state and the form Q.  TAU1: tau_f = tau_T = 1 (f, h are not read); then
// wscale multiplies every output (the FP16 storage scale).  SOURCES = false
// keeps the equilibria alone.
template <bool TAU1, bool SOURCES, class L, class R>
__device__ __forceinline__ void core_emit(const KConst<R>& k, const Cell<L>& c, const CoreState<L>& s, L Qxx, L Qyy,
                                          L Q2, const L* f, const L* h, L* fo, L* ho, R wscale) {
    const L w1 = lset<L>(wscale * (R(1) / R(9)));
    const L nthird = lset<L>(R(-1) / R(3));
    // out_i, out_j = w (e +- d) of two opposite directions.  The smaller of
    // the two parts is scaled by w first, so that each output is rounded once
    // at its own size: in the flow e ~ u^2 < d ~ u, in the temperature d < e.
    auto put_f = [&](int i, int j, const L& w, const L& e, const L& d) {
        const L b = lmul(w, e), n = lneg(w);
        fo[i] = lfma(w, d, TAU1 ? b : lfma(lset<L>(k.omf), f[i], b));
        fo[j] = lfma(n, d, TAU1 ? b : lfma(lset<L>(k.omf), f[j], b));
    };
    {
        const L tr = ladd(Qxx, Qyy);
        const L E = lfma(nthird, tr, lmul(lset<L>(k.fA_ep), s.ep));
        const L Ed = ladd(E, tr);
        const L fu = lset<L>(k.f_cu), fF = lset<L>(k.f_cF);
        const L Dx = SOURCES ? lfma(fu, s.ux, lmul(fF, s.Fx)) : lmul(fu, s.ux);
        const L Dy = SOURCES ? lfma(fu, s.uy, lmul(fF, s.Fy)) : lmul(fu, s.uy);
        // the flow's own diagonal weight, rounded to nearest: 2 w_1 + 4 w_5 is
        // then within 7.5e-9 of 1/3, which scales the momentum in each step
        // (w_diag, fitted to the sum of all nine, is 1.5e-8 off)
        const L w5 = lset<L>(wscale * (R(1) / R(36)));
        put_f(1, 3, w1, ladd(E, Qxx), Dx);
        put_f(2, 4, w1, ladd(E, Qyy), Dy);
        put_f(5, 7, w5, ladd(Ed, Q2), SOURCES ? ladd(Dx, Dy) : lfma(fu, s.uy, Dx));
        put_f(6, 8, w5, lsub(Ed, Q2), SOURCES ? lsub(Dy, Dx) : lfma(lset<L>(-k.f_cu), s.ux, Dy));
    }
    {
        // even part: sigma theta plus small terms, summed among themselves first
        const L T = s.T, Tep = lmul(T, s.ep);
        const L th = lmul(lset<L>(k.h_sig), s.th);
        const L kc = lmul(c.kc, T);
        const L kx = lmul(kc, s.ux), ky = lmul(kc, s.uy);
        const L tr = lfma(kx, s.ux, lmul(ky, s.uy));
        const L m0 = SOURCES ? lfma(nthird, tr, lset<L>(k.h_kQ)) : lmul(nthird, tr);
        // h + (w sum h - h)/tau + w (small +- d): the difference is small, so
        // the output is rounded once at its own size here too; sigma theta =
        // sum h + Q/2, and what the sum in R misses joins the small terms
        const L itT = lset<L>(R(1) - k.omT);
        L tr0, m1 = m0;
        if constexpr (!TAU1) {
            tr0 = core_hsum(h);
            m1 = lfma(itT, ladd(core_hsum_rest(h), lset<L>(k.half_Q)), m0);
        }
        const L m = lfma(lset<L>(k.h_pT), Tep, m1);
        const L md = SOURCES ? ladd(m, tr) : lfma(lset<L>(R(1)), tr, m);
        L Vx, Vy;
        if constexpr (SOURCES) {
            const L K = lfma(lset<L>(k.h_u3), T, lfma(c.ug, lfma(s.ux, s.gx, lmul(s.uy, s.gy)), lset<L>(k.h_uQ)));
            const L hg = lfma(lset<L>(k.h_Wr), s.ep, lset<L>(k.h_g)), hT = lmul(lset<L>(k.h_W), T);
            Vx = lfma(K, s.ux, lfma(hg, s.gx, lmul(hT, s.Fx)));
            Vy = lfma(K, s.uy, lfma(hg, s.gy, lmul(hT, s.Fy)));
        } else {
            const L K = lmul(lset<L>(k.h_u3), T), hg = lset<L>(k.h_g);
            Vx = lfma(K, s.ux, lmul(hg, s.gx));
            Vy = lfma(K, s.uy, lmul(hg, s.gy));
        }
        const L w5 = lset<L>(wscale * w_diag<R>());
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
        put_h(1, 3, w1, lfma(kx, s.ux, m), Vx);
        put_h(2, 4, w1, lfma(ky, s.uy, m), Vy);
        const L k2 = lmul(lset<L>(R(2)), kx);
        put_h(5, 7, w5, lfma(k2, s.uy, md), ladd(Vx, Vy));
        put_h(6, 8, w5, lfma(lneg(k2), s.uy, md), lsub(Vy, Vx));
        const L w0 = lset<L>(wscale * (R(4) / R(9)));
        const L pT = lset<L>(wscale * k.h0_pT);
        if constexpr (TAU1) ho[0] = lfma(w0, th, lfma(w0, m0, lmul(pT, Tep)));
        else ho[0] = ladd(h[0], lfma(itT, lfma(w0, tr0, lneg(h[0])), lfma(w0, m1, lmul(pT, Tep))));
    }
}

// Interior node: moments, then the collision.  The rest direction's thermal
// value is finite only if T and u are, so it stands for both.
template <bool TAU1, class L, class R>
__device__ __forceinline__ void core_interior(const KConst<R>& k, const Cell<L>& c, L eay, const L* f, const L* h,
                                              L* fo, L* ho, R wscale = R(1)) {
    const CoreState<L> s = core_moments(k, c, eay, f, h);
    L Qxx, Qyy, Q2;
    core_form(k, c, s, Qxx, Qyy, Q2);
    core_emit<TAU1, true>(k, c, s, Qxx, Qyy, Q2, f, h, fo, ho, wscale);
    if (!lfinite(ho[0])) atomicOr(k.flag, 1);
}

// Wall node at tau_f = tau_T = 1 (Sec. 3.4): there the extrapolated
// non-equilibrium part carries the factor 1 - 1/tau = 0, so the node is the
// collision of its boundary state b alone.  s, S: state and shear rate of
// x_f (on entry s; b on return), cs / cb: constants of x_f and of the node,
// thff: T(x_ff) - T0, thb: the Dirichlet T_b - T0 where `given`.
template <class L, class R>
__device__ __forceinline__ void core_boundary(const KConst<R>& k, const Cell<L>& cs, const Cell<L>& cb, L eay_b,
                                              R ubx, R uby, R ubm, bool given, bool fixgx, bool fixgy, R thb, L thff,
                                              CoreState<L>& s) {
    s.ux = lset<L>(ubx);
    s.uy = lset<L>(uby);
    if (given) {
        s.th = lset<L>(thb);
    } else {
        // Eq. (TNEESApGra) with zero normal gradient
        s.th = lmul(lset<L>(R(1) / R(3)), lfma(lset<L>(R(4)), s.th, lneg(thff)));
        if (fixgx) s.gx = lset<L>(R(0));
        if (fixgy) s.gy = lset<L>(R(0));
    }
    s.T = ladd(lset<L>(k.T0), s.th);
    // p(x_f) at the wall node's own porosity
    if (k.eps_field) s.ep = lmul(lmul(s.ep, cs.ie), cb.eps);
    const L nd = lfma(cb.nFK, lset<L>(ubm), cb.nnuK);
    s.Fx = lfma(nd, s.ux, cb.eax);
    s.Fy = lfma(nd, s.uy, lfma(cb.eg, s.th, eay_b));
}

}  // namespace lbm
