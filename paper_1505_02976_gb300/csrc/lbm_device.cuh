// lbm_device.cuh -- per-node arithmetic of the modified LBGK step (device side).
//
// One node of one time step, in the order the paper defines it:
//   pull-stream f_i, g_i from x - c_i                      (Eq. LBEeq, streaming of Sec. 3.2)
//   T from sigma T = sum g + Q/2                            (Sec. 3.2)
//   G = g beta (T - T0) j + a; v; u from the quadratic solve (Sec. 3.1)
//   F = -eps nu/K u - eps F_eps/sqrt(K) |u| u + eps G        (Eq. ForceEq)
//   p from sum_{i!=0} f_i, F_0 and s_0                       (Sec. 3.1, Appendix A)
//   S from the non-equilibrium second moment                 (Eq. ShearEqCom)
//   grad T from the 2x2 system M grad T = N                  (Eqs. TeEqCom-MatrN)
//   collide f and g                                          (Eqs. LBEeq, TEqColli)
// Wall nodes are rebuilt by non-equilibrium extrapolation from x_f (Sec. 3.4).
//
// The tensor contractions are expanded in closed form for D2Q9 (c_s^2 = 1/3):
//   s_i  = w_i [3 cu + 4.5 cu^2/eps - 1.5 |u|^2/eps]
//   r_i  = 1.5 w_i A [cx^2 Sxx + 2 cx cy Sxy + cy^2 Syy - (Sxx + Syy)/3]
//   F_i  = w_i rho0 (1 - 1/2tau_f) [3 cF + 9 cu cF/eps - 3 u.F/eps]
//   P_i  = w_i (1 - 1/2tau_T) [3 c.(T F + eps p grad T/rho0) + 3 (1/eps - 1/sigma) cu (u.grad T)]
//   Q_i  = w_i (1 - 1/2tau_T) (1 + 3 cu/sigma) Q
// and the moments the local schemes need use the closed-form equilibrium
// moments (Appendix A, Eq. EqZEqu; Sec. 3.2, Eq. MeOtEq):
//   sum c c f^{e(0)} = eps p I + rho0 u u / eps,  sum c g^{e(0)} = T u.
//
// Storage: flow populations f_1..f_8 as they are (f_0 is never read: p uses
// sum_{i!=0} f_i, u uses sum c_i f_i, S uses sum c c (f - f^{e(0)})), thermal
// populations as deviations h_i = g_i - w_i sigma T0 from the rest state.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

#include <type_traits>

#include "lbm_half.cuh"

namespace lbm {

// D2Q9 in the paper's order (Sec. 3.1).
__host__ __device__ constexpr int cx_of(int i) {
    return i == 1 || i == 5 || i == 8 ? 1 : (i == 3 || i == 6 || i == 7 ? -1 : 0);
}
__host__ __device__ constexpr int cy_of(int i) {
    return i == 2 || i == 5 || i == 6 ? 1 : (i == 4 || i == 7 || i == 8 ? -1 : 0);
}
// Weight of the diagonal directions, 1/36.  In FP32, 1/9 and 4/9 round to
// exactly 4 and 16 times the rounded 1/36, so the nine rounded weights would
// sum to 36 fl(1/36) = 1 + 7.45e-9: every step would scale the zeroth
// moments (T - T0, and the pressure) by that factor, a bias that builds up
// to ~1e-4 of the temperature over 1e5 steps.  The FP32 value is therefore
// one unit in the last place below fl(1/36) (2^-29 smaller), which makes the
// FP32 weights sum to exactly 1; the second moment moves by 1.5e-8 relative
// (a constant change of the viscosity of that size, which does not build up).
template <class R>
__host__ __device__ constexpr R w_diag() { return R(1) / R(36); }
template <>
__host__ __device__ constexpr float w_diag<float>() { return 0x1.c71c7p-6f; }

template <class R>
__host__ __device__ constexpr R w_of(int i) {
    return i == 0 ? R(4) / R(9) : (i <= 4 ? R(1) / R(9) : w_diag<R>());
}

enum : int { BC_PERIODIC = 0, BC_DIRICHLET = 1, BC_ADIABATIC = 2 };
enum : int { SW = 0, SE = 1, SS = 2, SN = 3 };

// Porosity-dependent constants of the node update (lbm_core.cuh): e the
// porosity, itf, itT = 1/tau, a = 1.5 itf rho0 A invD the share of S in Q.
template <class V>
struct Cell {
    V eps, ie, elo;    // e, 1/e, and 1/ie - e (what rounding left of e (1/e) = 1)
    V eg, eax, heax;   // e g beta, e a_x, e a_x / 2
    V c0, c0sq, c1;    // quadratic solve (Sec. 3.1)
    V nnuK, nFK;       // - e nu/K, - e F_e/sqrt(K)
    V e2, e3, e3_lo;   // e p = e1 sum f + e2 u.F + e3 |u|^2; e3_lo: what rounding e3 left
    V re;              // rho0 / e
    V qu, qF;          // of u u and u F in Q, S folded in: cu2 - a re, cuF + a re
    V cu2, cuF;        // the same with S apart: 4.5 itf rho0/e, 9 rho0 (1 - 1/2tau_f)/e
    V b, nb, ug, kc;   // (1/e - 1/sigma)/2, -b, 6 (1 - 1/2tau_T) b, 4.5 itT/e
};

// Constants of one run in the compute type R (filled on the host).
template <class R>
struct KConst {
    int nx, ny, pitch;     // pitch: elements per stored row
    int bc[4];
    long long plane;       // elements per stored plane (ny * pitch)
    R rho0, eps, inv_eps, sigma, inv_sigma;
    R omf, omT;            // 1 - 1/tau
    R tau_f, kf, kT;       // kf, kT = 1 - 1/(2 tau)
    R A, B, T0, gbeta, ax, ay, Q;
    R e_nuK, e_FK;         // eps nu / K, eps F_eps / sqrt(K)
    R c0, c0sq, c1;
    R p_pref;              // c_s^2 / (eps (1 - w_0)) = 3 / (5 eps)
    R invD;                // 1 / (c_s^2 rho0 (A - tau_f))
    R a_const;             // c_s^2 sigma (B - tau_T)
    R bcoef;               // (1/eps - 1/sigma) / 2
    R sT0;                 // sigma T0
    R T_bc[4];
    R u_bc[4][2];
    float scale;           // FP16 storage: stored value = population / scale
    float inv_scale;       // 1 / scale (a power of two)
    int* flag;             // non-finite flag (device)
    int plane32;           // plane stride as a 32-bit offset (17 planes < 2^31 elements)
    // porosity field (nullptr: uniform eps).  With a field, K follows the
    // Kozeny-Carman form of the Ergun permeability, K(eps) = K_ref r(eps) with
    // r(eps) = [eps^3 / (1 - eps)^2] / [eps_ref^3 / (1 - eps_ref)^2].
    const R* eps_field;    // [ny][nx]
    R kc_inv_ref;          // (1 - eps_ref)^2 / eps_ref^3
    R nu_over_Kref;        // nu / K_ref
    R inv_sqrt_Kref;       // 1 / sqrt(K_ref)
    R p_pref_eps;          // c_s^2 / (1 - w_0)
    int da_inf, forch;
    const R* ay_row;       // extra external acceleration a_y per row, or nullptr
    // constants of the node update (lbm_core.cuh): those of the uniform
    // porosity, and the factors that give a porosity field's
    Cell<R> cell;
    R inv_rho0, hq_sigma, half_Q, eay, half_ax;      // 1/rho0, Q/(2 sigma), Q/2, eps a_y, a_x/2
    R nnuK_q2, nnuK_0, nFK_q, e1, e1_lo, e2_ie, e3_ie, qu_ie, qF_ie, cu2_ie, cuF_ie, b_0, ug_b, kc_ie;
    R a_ep, aS, aS2, f_ScS, f_ScS2, fA_ep, f_cu, f_cF;
    R h_sig, h_kQ, h_pT, h0_pT, h_u3, h_uQ, h_g, h_W, h_Wr;
    R u_abs[4];            // |u_bc| per side
    // nodes at the end of a staged step's sweep whose stores ask L2 to keep
    // them (evict-last hint): the next step reads those rows first (0: none)
    long long l2_hot;
};

// Population storage conversion.
template <class S, class R>
__device__ __forceinline__ R load_pop(const S* p, float) { return R(*p); }
template <>
__device__ __forceinline__ float load_pop<__half, float>(const __half* p, float scale) {
    return __half2float(*p) * scale;
}
template <class S, class R>
__device__ __forceinline__ void store_pop(S* p, R v, float) { *p = S(v); }
template <>
__device__ __forceinline__ void store_pop<__half, float>(__half* p, float v, float scale) {
    *p = __float2half_rn(v / scale);
}

// Store of the 17 post-collision values of one node; FP16 storage rounds
// stochastically (dither != nullptr) or to nearest (lbm_half.cuh).
// evict_last (FP32 storage): the stores carry an L2 evict-last policy.
template <class S, class R>
__device__ __forceinline__ void store_planes(S* __restrict__ d, long long pl, const R* fo, const R* ho,
                                             float inv_scale, Dither* dither, bool evict_last = false) {
    if constexpr (std::is_same<S, __half>::value) {
        store_planes_half<R>(d, pl, fo, ho, inv_scale, dither);
    } else {
        if constexpr (std::is_same<S, float>::value) {
            if (evict_last) {
                uint64_t pol;
                asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
#pragma unroll
                for (int i = 1; i < 9; ++i)
                    asm volatile("st.global.L2::cache_hint.f32 [%0], %1, %2;" ::"l"(d + (i - 1) * pl),
                                 "f"(float(fo[i])), "l"(pol) : "memory");
#pragma unroll
                for (int i = 0; i < 9; ++i)
                    asm volatile("st.global.L2::cache_hint.f32 [%0], %1, %2;" ::"l"(d + (8 + i) * pl),
                                 "f"(float(ho[i])), "l"(pol) : "memory");
                return;
            }
        }
#pragma unroll
        for (int i = 1; i < 9; ++i) d[(i - 1) * pl] = S(fo[i]);
#pragma unroll
        for (int i = 0; i < 9; ++i) d[(8 + i) * pl] = S(ho[i]);
    }
}

// Plane k of the stored state: k = 0..7 hold f_1..f_8, k = 8..16 hold h_0..h_8.
constexpr int NPLANES = 17;

template <class R>
struct Pops {
    R f[9];  // f[0] unused
    R h[9];
};

// Role of node (x, y): interior, or a wall node with its NEES neighbours.
struct WallInfo {
    int wall;       // 0 interior
    int xs, ys;     // node whose post-streaming state is used (x itself, or x_f)
    int xff, yff;   // x_ff for the Neumann extrapolation
    int tside;      // side whose Dirichlet T applies, -1: adiabatic
    int uside;      // side whose wall velocity applies
    int fixgx, fixgy;
};

template <class R>
__device__ __forceinline__ WallInfo classify(const KConst<R>& k, int x, int y) {
    WallInfo w;
    const bool onW = x == 0 && k.bc[SW] != BC_PERIODIC;
    const bool onE = x == k.nx - 1 && k.bc[SE] != BC_PERIODIC;
    const bool onS = y == 0 && k.bc[SS] != BC_PERIODIC;
    const bool onN = y == k.ny - 1 && k.bc[SN] != BC_PERIODIC;
    w.wall = onW || onE || onS || onN;
    const int dx = onW ? 1 : (onE ? -1 : 0);
    const int dy = onS ? 1 : (onN ? -1 : 0);
    w.xs = x + dx;
    w.ys = y + dy;
    w.xff = x + 2 * dx;
    w.yff = y + 2 * dy;
    const int xsd = onW ? SW : (onE ? SE : -1);
    const int ysd = onS ? SS : (onN ? SN : -1);
    w.tside = -1;
    if (xsd >= 0 && k.bc[xsd] == BC_DIRICHLET) w.tside = xsd;
    else if (ysd >= 0 && k.bc[ysd] == BC_DIRICHLET) w.tside = ysd;
    w.uside = xsd >= 0 ? xsd : (ysd >= 0 ? ysd : 0);
    w.fixgx = xsd >= 0;
    w.fixgy = ysd >= 0;
    return w;
}

template <class R>
__device__ __forceinline__ bool is_wall(const KConst<R>& k, int x, int y) {
    return (x == 0 && k.bc[SW] != BC_PERIODIC) || (x == k.nx - 1 && k.bc[SE] != BC_PERIODIC) ||
           (y == 0 && k.bc[SS] != BC_PERIODIC) || (y == k.ny - 1 && k.bc[SN] != BC_PERIODIC);
}

// Column x is a W or E wall column.
template <class R>
__device__ __forceinline__ bool is_wall_x(const KConst<R>& k, int x) {
    return (x == 0 && k.bc[SW] != BC_PERIODIC) || (x == k.nx - 1 && k.bc[SE] != BC_PERIODIC);
}

// Post-streaming populations of node (x, y): f_i and g_i pulled from x - c_i.
template <class R, class S>
__device__ __forceinline__ void pull(const KConst<R>& k, const S* __restrict__ src, int x, int y,
                                     Pops<R>& P) {
    const int xm = x == 0 ? k.nx - 1 : x - 1;
    const int xp = x == k.nx - 1 ? 0 : x + 1;
    const int ym = y == 0 ? k.ny - 1 : y - 1;
    const int yp = y == k.ny - 1 ? 0 : y + 1;
    const long long r0 = (long long)y * k.pitch, rm = (long long)ym * k.pitch,
                    rp = (long long)yp * k.pitch;
    // source of direction i is x - c_i
    const long long at[9] = {r0 + x, r0 + xm, rm + x, r0 + xp, rp + x,
                             rm + xm, rm + xp, rp + xp, rp + xm};
    const float sc = k.scale;
#pragma unroll
    for (int i = 1; i < 9; ++i) P.f[i] = load_pop<S, R>(src + (long long)(i - 1) * k.plane + at[i], sc);
#pragma unroll
    for (int i = 0; i < 9; ++i) P.h[i] = load_pop<S, R>(src + (long long)(8 + i) * k.plane + at[i], sc);
    P.f[0] = R(0);
}

// Sum of the thermal deviations pulled into (x, y), accumulated in Acc (for T alone).
template <class Acc, class R, class S>
__device__ __forceinline__ Acc pull_hsum(const KConst<R>& k, const S* __restrict__ src, int x, int y) {
    const int xm = x == 0 ? k.nx - 1 : x - 1;
    const int xp = x == k.nx - 1 ? 0 : x + 1;
    const int ym = y == 0 ? k.ny - 1 : y - 1;
    const int yp = y == k.ny - 1 ? 0 : y + 1;
    const long long r0 = (long long)y * k.pitch, rm = (long long)ym * k.pitch,
                    rp = (long long)yp * k.pitch;
    const long long at[9] = {r0 + x, r0 + xm, rm + x, r0 + xp, rp + x,
                             rm + xm, rm + xp, rp + xp, rp + xm};
    Acc s = Acc(0);
#pragma unroll
    for (int i = 0; i < 9; ++i) s += Acc(load_pop<S, R>(src + (long long)(8 + i) * k.plane + at[i], k.scale));
    return s;
}

// Porosity-dependent constants of one node, and the y-component of the
// external acceleration a at its row.
template <class V>
struct CellC {
    V eps, inv_eps, e_nuK, e_FK, c0, c0sq, c1, p_pref, bcoef, ay;
};

// a_y at row y: the uniform a_y plus the optional per-row profile.
template <class R>
__device__ __forceinline__ R row_ay(const KConst<R>& k, int y) {
    return k.ay_row ? k.ay + k.ay_row[y] : k.ay;
}

template <class R>
__device__ __forceinline__ R node_eps(const KConst<R>& k, int x, int y) {
    return k.eps_field ? k.eps_field[(long long)y * k.nx + x] : k.eps;
}

// Constants at porosity eps: the run's own constants for a uniform porosity,
// else from the Kozeny-Carman permeability K(eps) and the Ergun F_eps(eps)
// (Sec. 2): e_nuK = eps nu/K, e_FK = eps F_eps/sqrt(K), c0 = (1 + e_nuK/2)/2,
// c1 = e_FK/2 (Sec. 3.1).
template <class R, class V>
__device__ __forceinline__ CellC<V> cell_consts(const KConst<R>& k, V eps) {
    CellC<V> c;
    if (!k.eps_field) {
        c.eps = V(k.eps);
        c.inv_eps = V(k.inv_eps);
        c.e_nuK = V(k.e_nuK);
        c.e_FK = V(k.e_FK);
        c.c0 = V(k.c0);
        c.c0sq = V(k.c0sq);
        c.c1 = V(k.c1);
        c.p_pref = V(k.p_pref);
        c.bcoef = V(k.bcoef);
        c.ay = V(k.ay);
        return c;
    }
    c.eps = eps;
    c.inv_eps = R(1) / eps;
    if (k.da_inf) {
        c.e_nuK = V(R(0));
        c.e_FK = V(R(0));
    } else {
        const V om = R(1) - eps;
        const V ratio = eps * eps * eps / (om * om) * k.kc_inv_ref;  // K / K_ref
        c.e_nuK = eps * k.nu_over_Kref / ratio;
        if (k.forch) {
            const V Feps = R(1.75) / sqrt(R(150) * eps * eps * eps);
            c.e_FK = eps * Feps * k.inv_sqrt_Kref / sqrt(ratio);
        } else {
            c.e_FK = V(R(0));
        }
    }
    c.c0 = R(0.5) + R(0.25) * c.e_nuK;
    c.c0sq = c.c0 * c.c0;
    c.c1 = R(0.5) * c.e_FK;
    c.p_pref = k.p_pref_eps * c.inv_eps;
    c.bcoef = R(0.5) * (c.inv_eps - k.inv_sigma);
    c.ay = V(k.ay);
    return c;
}

template <class V>
struct State {
    V th;               // T - T0
    V ux, uy, Fx, Fy;   // velocity, total force
    V p;
    V Sxx, Sxy, Syy;    // shear rate
    V gx, gy;           // grad T
};

// Moments of one node from its post-streaming populations (f[1..8], h[0..8]).
template <class R, class V>
__device__ __forceinline__ State<V> node_moments(const KConst<R>& k, const CellC<V>& c, const V* f,
                                                 const V* h) {
    State<V> s;
    // sigma T = sum g + Q/2, with sum g = sum h + sigma T0
    const V sh = h[0] + h[1] + h[2] + h[3] + h[4] + h[5] + h[6] + h[7] + h[8];
    s.th = (sh + R(0.5) * k.Q) * k.inv_sigma;
    const V T = k.T0 + s.th;
    // flow moments
    const V sf = f[1] + f[2] + f[3] + f[4] + f[5] + f[6] + f[7] + f[8];
    const V mx = (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7]);
    const V my = (f[2] - f[4]) + (f[5] - f[8]) + (f[6] - f[7]);
    const V d58 = f[5] + f[6] + f[7] + f[8];
    const V Pxx = f[1] + f[3] + d58;
    const V Pyy = f[2] + f[4] + d58;
    const V Pxy = (f[5] + f[7]) - (f[6] + f[8]);
    // buoyancy, temporary velocity, quadratic solve
    const R Gx = k.ax;
    const V Gy = k.gbeta * s.th + c.ay;
    const V vx = mx * k.inv_rho0 + R(0.5) * c.eps * Gx;
    const V vy = my * k.inv_rho0 + R(0.5) * c.eps * Gy;
    const V vmag = sqrt(vx * vx + vy * vy);
    const V den = c.c0 + sqrt(c.c0sq + c.c1 * vmag);
    s.ux = vx / den;
    s.uy = vy / den;
    const V uu = s.ux * s.ux + s.uy * s.uy;
    const V umag = sqrt(uu);
    const V drag = c.e_nuK + c.e_FK * umag;
    s.Fx = c.eps * Gx - drag * s.ux;
    s.Fy = c.eps * Gy - drag * s.uy;
    const V uF = s.ux * s.Fx + s.uy * s.Fy;
    // p = c_s^2/(eps (1-w0)) [sum_{i!=0} f + tau_f F_0 + rho0 s_0],
    // F_0 = -3 w0 rho0 kf u.F/eps, s_0 = -1.5 w0 |u|^2/eps, w0 = 4/9
    const V F0 = -(R(4) / R(3)) * k.rho0 * k.kf * uF * c.inv_eps;
    const V s0 = -(R(2) / R(3)) * uu * c.inv_eps;
    s.p = c.p_pref * (sf + k.tau_f * F0 + k.rho0 * s0);
    // S = [Pi - eps p I - rho0 u u/eps + (rho0/2)(uF + Fu)/eps] / (c_s^2 rho0 (A - tau_f))
    const V re = k.rho0 * c.inv_eps;
    const V ep = c.eps * s.p;
    s.Sxx = (Pxx - ep - re * s.ux * s.ux + re * s.ux * s.Fx) * k.invD;
    s.Syy = (Pyy - ep - re * s.uy * s.uy + re * s.uy * s.Fy) * k.invD;
    s.Sxy = (Pxy - re * s.ux * s.uy + R(0.5) * re * (s.ux * s.Fy + s.Fx * s.uy)) * k.invD;
    // N = sum c (g - g^{e(0)}) + (T F + u Q/sigma)/2 with sum c g^{e(0)} = T u
    const V nx_ = (h[1] - h[3]) + (h[5] - h[6]) + (h[8] - h[7]);
    const V ny_ = (h[2] - h[4]) + (h[5] - h[8]) + (h[6] - h[7]);
    const R qs = R(0.5) * k.Q * k.inv_sigma;
    const V Nx = nx_ - T * s.ux + R(0.5) * T * s.Fx + qs * s.ux;
    const V Ny = ny_ - T * s.uy + R(0.5) * T * s.Fy + qs * s.uy;
    // M = a I - b u u^T, a = -eps p/(2 rho0) + c_s^2 sigma (B - tau_T),
    // b = (1/eps - 1/sigma)/2; M^{-1} N = (N + b u (u.N)/(a - b|u|^2)) / a
    const V a = k.a_const - R(0.5) * ep * k.inv_rho0;
    const V uN = s.ux * Nx + s.uy * Ny;
    const V t = c.bcoef * uN / (a - c.bcoef * uu);
    const V ia = R(1) / a;
    s.gx = (Nx + t * s.ux) * ia;
    s.gy = (Ny + t * s.uy) * ia;
    return s;
}

// Equilibria and source terms of one state, direction by direction.
template <class V>
struct EqTerms {
    V fe[9];   // f^eq_i, i = 1..8 (index 0 unused)
    V Fi[9];   // forcing term F_i, i = 1..8
    V he[9];   // g^eq_i - w_i sigma T0
    V PQ[9];   // P_i + Q_i
};

template <class R, class V>
__device__ __forceinline__ void eq_terms(const KConst<R>& k, const CellC<V>& c, const State<V>& s,
                                         EqTerms<V>& e) {
    const V T = k.T0 + s.th;
    const V uu = s.ux * s.ux + s.uy * s.uy;
    const V ie = c.inv_eps;
    const V flow_c = R(3) * c.eps * s.p - R(1.5) * k.rho0 * uu * ie - R(0.5) * k.rho0 * k.A * (s.Sxx + s.Syy);
    const V uF = s.ux * s.Fx + s.uy * s.Fy;
    const V force_c = -R(3) * uF * ie;
    const V pT = R(3) * T * c.eps * s.p * k.inv_rho0;   // 3 T eps p / rho0
    const V ug = s.ux * s.gx + s.uy * s.gy;
    const V Wx = T * s.Fx + c.eps * s.p * s.gx * k.inv_rho0;
    const V Wy = T * s.Fy + c.eps * s.p * s.gy * k.inv_rho0;
    const V therm_c = k.sigma * s.th - R(1.5) * T * uu * ie;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const R cx = R(cx_of(i)), cy = R(cy_of(i));
        const R w = w_of<R>(i);
        const V cu = cx * s.ux + cy * s.uy;
        const V cF = cx * s.Fx + cy * s.Fy;
        if (i > 0) {
            const V ScS = cx * cx * s.Sxx + R(2) * cx * cy * s.Sxy + cy * cy * s.Syy;
            e.fe[i] = w * (flow_c + k.rho0 * (R(3) * cu + R(4.5) * cu * cu * ie) + R(1.5) * k.rho0 * k.A * ScS);
            e.Fi[i] = w * k.rho0 * k.kf * (R(3) * cF + R(9) * cu * cF * ie + force_c);
        } else {
            e.fe[0] = V(R(0));
            e.Fi[0] = V(R(0));
        }
        const V cg = cx * s.gx + cy * s.gy;
        // varpi_0 = -5/9 = -(1 - w0); varpi_i = w_i otherwise
        const V pv = (i == 0) ? -(R(5) / R(9)) * pT : w * pT;
        e.he[i] = w * (therm_c + T * (R(3) * cu + R(4.5) * cu * cu * ie) + k.sigma * k.B * cg) + pv;
        const V cW = cx * Wx + cy * Wy;
        e.PQ[i] = w * k.kT * (R(3) * cW + R(6) * c.bcoef * cu * ug + (R(1) + R(3) * cu * k.inv_sigma) * k.Q);
    }
}

// Boundary state of a wall node (Sec. 3.4): u_b, T_b, p(x_f), S(x_f),
// grad T_b, and F at (u_b, T_b) with the wall node's own porosity (cb).
// thff is T(x_ff) - T0 (adiabatic walls), thb the Dirichlet T_b - T0.
template <class R, class V>
__device__ __forceinline__ State<V> wall_state(const KConst<R>& k, const CellC<V>& cb, const WallInfo& w,
                                               const State<V>& sf, V thff, V thb) {
    State<V> b = sf;
    b.ux = V(k.u_bc[w.uside][0]);
    b.uy = V(k.u_bc[w.uside][1]);
    if (w.tside >= 0) {
        b.th = thb;
    } else {
        // Eq. (TNEESApGra) with zero normal gradient
        if (w.fixgx) b.gx = V(R(0));
        if (w.fixgy) b.gy = V(R(0));
        b.th = (R(4) * sf.th - thff) * (R(1) / R(3));
    }
    const V umag = sqrt(b.ux * b.ux + b.uy * b.uy);
    const V drag = cb.e_nuK + cb.e_FK * umag;
    b.Fx = cb.eps * k.ax - drag * b.ux;
    b.Fy = cb.eps * (k.gbeta * b.th + cb.ay) - drag * b.uy;
    return b;
}

// Planes of the moment state (tau = 1 storage): p, u, S, T - T0, grad T.
enum MomentPlane { MP = 0, MUX, MUY, MSXX, MSYY, MSXY, MTH, MGX, MGY };
constexpr int kMPlanes = 9;

}  // namespace lbm
