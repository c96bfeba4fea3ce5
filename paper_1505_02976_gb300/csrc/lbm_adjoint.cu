// lbm_adjoint.cu -- discrete adjoint of the fused step (lbm_adjoint).
//
// Loss: the mean Nusselt number on one wall after n steps (Eq. Eq:AvNuss),
// as a function of the porosity field and of the Dirichlet wall
// temperatures.  The step maps the post-collision state s_n to s_{n+1};
// node x of s_{n+1} depends on the 17 populations it pulls from its source
// node (x itself, or x_f for a wall node), on T(x_ff) for adiabatic walls,
// on the porosity at the source and at x, and on the Dirichlet T_b.  The
// adjoint runs the steps backwards, one launch a step (k_adj_step): the thread
// of interior node s pulls its 17 values of the state again, and takes the
// adjoint of everything computed from them -- its own collision and, beside a
// wall, the collisions of the up to three wall nodes whose x_f it is -- back
// through the moments to the 17 pulled values (reverse mode, by hand: about
// three times the operations of the step).  The transpose of pull streaming
// is then a store of each adjoint at the place it was pulled from: every
// place is pulled by at most one interior node, so no two threads write the
// same word and the result does not depend on their order.
// A run whose states fit 256 MB keeps them all; a longer one keeps checkpoints
// every ceil(sqrt(n)) steps and recomputes the states between them.
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <string>
#include <type_traits>
#include <vector>

#include "lbm_core.cuh"
#include "lbm_handle.h"
#include "lbm_host.h"
#include "lbm_internal.h"

namespace lbm {

constexpr int kAdjBlock = 128;

template <class R>
__device__ __forceinline__ long long at_of(const KConst<R>& k, int x, int y) { return (long long)y * k.pitch + x; }

// Adjoint of the state a collision is computed from, T and p folded into th
// and ep.
template <class R>
struct StateBar {
    R th, ux, uy, Fx, Fy, ep, Sxx, Syy, Sxy, gx, gy;
};
// Adjoint of a node's porosity constants: e itself, 1/e, and the drag
// coefficients a1 = e nu/K, a2 = e F_e/sqrt(K).
template <class R>
struct CellBar {
    R e, ie, a1, a2;
};

// What the backward pass needs of a node's moments (node_moments' names).
template <class R>
struct AdjState {
    R e, ie, a1, a2, c0, c1;           // porosity and its constants
    R th, T, Gy, vx, vy, vm, rs, iden; // rs: sqrt(c0^2 + c1 |v|)
    R ux, uy, um, drag, Fx, Fy, uu, ep;
    R Sxx, Syy, Sxy, Px, Py, Nx, Ny, ia, id, t, gx, gy;
};

// Collision adjoint: adds to B and C what the outputs' adjoints lf (flow) and
// lh (thermal) give for f^eq, g^eq of the state, scaled by sF, sT, and, with
// SOURCES, for F_i, P_i + Q_i (lbm_core.cuh: core_emit with S explicit).
template <bool SOURCES, class R>
__device__ __forceinline__ void emit_adjoint(const KConst<R>& k, R ie, R sF, R sT, R ux, R uy, R Fx, R Fy, R ep, R T,
                                             R gx, R gy, const R* lf, const R* lh, StateBar<R>& B, CellBar<R>& C) {
    const R w1 = R(1) / R(9), w5 = w_diag<R>(), w0 = R(4) / R(9);
    const R third = R(1) / R(3);
    {
        const R a1 = w1 * lf[1], a2 = w1 * lf[2], a3 = w1 * lf[3], a4 = w1 * lf[4];
        const R a5 = w5 * lf[5], a6 = w5 * lf[6], a7 = w5 * lf[7], a8 = w5 * lf[8];
        const R d = (a5 + a7) + (a6 + a8), x13 = a1 + a3, y24 = a2 + a4;
        const R LE = x13 + y24 + d;
        const R Qx = x13 + d - third * LE, Qy = y24 + d - third * LE, Q2 = (a5 + a7) - (a6 + a8);
        const R Dx = (a1 - a3) + (a5 - a7) + (a8 - a6), Dy = (a2 - a4) + (a5 - a7) + (a6 - a8);
        B.ep += R(3) * sF * LE;
        const R fS = R(1.5) * k.rho0 * k.A * sF;
        B.Sxx += fS * Qx;
        B.Syy += fS * Qy;
        B.Sxy += R(2) * fS * Q2;
        const R c2 = R(4.5) * k.rho0 * sF, cF = SOURCES ? R(9) * k.rho0 * k.kf : R(0);
        const R tx = ie * (R(2) * c2 * ux + cF * Fx), ty = ie * (R(2) * c2 * uy + cF * Fy);
        const R fu = R(3) * k.rho0 * sF;
        B.ux += Qx * tx + Q2 * ty + fu * Dx;
        B.uy += Qy * ty + Q2 * tx + fu * Dy;
        C.ie += c2 * (ux * ux * Qx + uy * uy * Qy + R(2) * ux * uy * Q2);
        if constexpr (SOURCES) {
            const R fF = R(3) * k.rho0 * k.kf;
            B.Fx += cF * ie * (ux * Qx + uy * Q2) + fF * Dx;
            B.Fy += cF * ie * (uy * Qy + ux * Q2) + fF * Dy;
            C.ie += cF * (ux * Fx * Qx + uy * Fy * Qy + (ux * Fy + uy * Fx) * Q2);
        }
    }
    {
        const R a1 = w1 * lh[1], a2 = w1 * lh[2], a3 = w1 * lh[3], a4 = w1 * lh[4];
        const R a5 = w5 * lh[5], a6 = w5 * lh[6], a7 = w5 * lh[7], a8 = w5 * lh[8];
        const R d = (a5 + a7) + (a6 + a8), x13 = a1 + a3, y24 = a2 + a4;
        const R M1 = x13 + y24 + d, M0 = M1 + w0 * lh[0];
        const R Bx = x13 + d, By = y24 + d, B2 = (a5 + a7) - (a6 + a8);
        const R Vx = (a1 - a3) + (a5 - a7) + (a8 - a6), Vy = (a2 - a4) + (a5 - a7) + (a6 - a8);
        const R uu = ux * ux + uy * uy;
        R Tb = R(0);  // adjoint of T
        B.th += k.sigma * sT * M0;
        const R kc = R(4.5) * sT;
        const R q = ux * ux * Bx + uy * uy * By + R(2) * ux * uy * B2 - third * uu * M0;
        Tb += kc * ie * q;
        C.ie += kc * T * q;
        const R kT2 = R(2) * kc * ie * T;
        B.ux += kT2 * (ux * Bx + uy * B2 - third * ux * M0);
        B.uy += kT2 * (uy * By + ux * B2 - third * uy * M0);
        const R Teb = sT * k.inv_rho0 * (R(3) * M1 - (R(5) / R(3)) * lh[0]);  // adjoint of T eps p
        Tb += ep * Teb;
        B.ep += T * Teb;
        const R Kb = ux * Vx + uy * Vy;
        R K = R(3) * sT * T, hg = k.sigma * k.B * sT;
        Tb += R(3) * sT * Kb;
        if constexpr (SOURCES) {
            const R W = R(3) * k.kT, b6 = R(6) * k.kT, ug = b6 * R(0.5) * (ie - k.inv_sigma), gu = ux * gx + uy * gy;
            K += ug * gu + W * k.Q * k.inv_sigma;
            hg += W * k.inv_rho0 * ep;
            B.ep += W * k.inv_rho0 * (gx * Vx + gy * Vy);
            B.Fx += W * T * Vx;
            B.Fy += W * T * Vy;
            Tb += W * (Fx * Vx + Fy * Vy);
            const R uk = ug * Kb;
            B.ux += uk * gx;
            B.uy += uk * gy;
            B.gx += uk * ux;
            B.gy += uk * uy;
            C.ie += R(0.5) * b6 * gu * Kb;
        }
        B.ux += K * Vx;
        B.uy += K * Vy;
        B.gx += hg * Vx;
        B.gy += hg * Vy;
        B.th += Tb;
    }
}

// Moments of an interior node (node_moments), every intermediate kept.
template <class R>
__device__ __forceinline__ AdjState<R> adjoint_state(const KConst<R>& k, R e, R ay, const R* f, const R* h) {
    AdjState<R> s;
    const Cell<R> c = k.eps_field ? field_cell<R>(k, e) : k.cell;
    s.e = c.eps;
    s.ie = c.ie;
    s.a1 = -c.nnuK;
    s.a2 = -c.nFK;
    s.c0 = c.c0;
    s.c1 = c.c1;
    s.th = (((h[1] + h[3]) + (h[2] + h[4])) + ((h[5] + h[7]) + (h[6] + h[8])) + h[0]) * k.inv_sigma + k.hq_sigma;
    s.T = k.T0 + s.th;
    const R s13 = f[1] + f[3], s24 = f[2] + f[4], s57 = f[5] + f[7], s68 = f[6] + f[8];
    const R d57 = f[5] - f[7], d86 = f[8] - f[6], d58 = s57 + s68;
    const R mx = (f[1] - f[3]) + (d57 + d86), my = (f[2] - f[4]) + (d57 - d86);
    s.Gy = k.gbeta * s.th + ay;
    s.vx = mx * k.inv_rho0 + R(0.5) * s.e * k.ax;
    s.vy = my * k.inv_rho0 + R(0.5) * s.e * s.Gy;
    s.vm = lsqrt(s.vx * s.vx + s.vy * s.vy);
    s.rs = lsqrt(c.c0sq + s.c1 * s.vm);
    s.iden = lrcp(s.c0 + s.rs);
    s.ux = s.vx * s.iden;
    s.uy = s.vy * s.iden;
    s.um = s.vm * s.iden;
    s.drag = s.a1 + s.a2 * s.um;
    s.Fx = s.e * k.ax - s.drag * s.ux;
    s.Fy = s.e * s.Gy - s.drag * s.uy;
    s.uu = s.ux * s.ux + s.uy * s.uy;
    const R uF = s.ux * s.Fx + s.uy * s.Fy;
    s.ep = k.e1 * (s13 + s24 + d58) + (c.e2 * uF + c.e3 * s.uu);
    s.Px = s13 + d58 - s.ep;
    s.Py = s24 + d58 - s.ep;
    const R Pxy = s57 - s68;
    const R dx = s.Fx - s.ux, dy = s.Fy - s.uy;
    s.Sxx = k.invD * (s.Px + c.re * s.ux * dx);
    s.Syy = k.invD * (s.Py + c.re * s.uy * dy);
    s.Sxy = k.invD * (Pxy + R(0.5) * c.re * (s.ux * dy + s.uy * dx));
    const R h57 = h[5] - h[7], h86 = h[8] - h[6];
    const R hx = (h[1] - h[3]) + (h57 + h86), hy = (h[2] - h[4]) + (h57 - h86);
    const R qT = k.hq_sigma - s.T;
    s.Nx = hx + s.ux * qT + R(0.5) * s.T * s.Fx;
    s.Ny = hy + s.uy * qT + R(0.5) * s.T * s.Fy;
    const R a = k.a_const + k.a_ep * s.ep, d = a - c.b * s.uu, r = lrcp(a * d);
    s.ia = d * r;
    s.id = a * r;
    s.t = c.b * (s.ux * s.Nx + s.uy * s.Ny) * r;
    s.gx = s.Nx * s.ia + s.t * s.ux;
    s.gy = s.Ny * s.ia + s.t * s.uy;
    return s;
}

// Adjoint of the moments: from B (adjoint of the state) to the adjoints of the
// moment sums M = (sum h, c h, sum f, c f, c c f), adding the porosity's to C.
template <class R>
struct SumsBar {
    R h0, hx, hy, f0, fx, fy, fxx, fyy, fxy;
};
template <class R>
__device__ __forceinline__ SumsBar<R> moments_adjoint(const KConst<R>& k, const AdjState<R>& s, StateBar<R> B,
                                                      CellBar<R>& C) {
    SumsBar<R> m;
    const R ux = s.ux, uy = s.uy, Fx = s.Fx, Fy = s.Fy;
    const R re = k.rho0 * s.ie, b = R(0.5) * (s.ie - k.inv_sigma);
    // S = [P + re (u F + F u)/2 - re u u]/D
    const R qxx = k.invD * B.Sxx, qyy = k.invD * B.Syy, qxy = k.invD * B.Sxy;
    const R dx = Fx - ux, dy = Fy - uy;
    m.fxy = qxy;
    C.ie += k.rho0 * (qxx * ux * dx + qyy * uy * dy + R(0.5) * qxy * (ux * dy + uy * dx));
    const R rx = re * qxx, ry = re * qyy, rxy = re * qxy;
    B.ux += rx * (Fx - R(2) * ux) + rxy * (R(0.5) * Fy - uy);
    B.uy += ry * (Fy - R(2) * uy) + rxy * (R(0.5) * Fx - ux);
    B.Fx += rx * ux + R(0.5) * rxy * uy;
    B.Fy += ry * uy + R(0.5) * rxy * ux;
    // grad T = N/a + t u, t = b u.N/(a d), d = a - b |u|^2, a = a_const + a_ep ep
    const R tb = ux * B.gx + uy * B.gy, ng = s.Nx * B.gx + s.Ny * B.gy;
    const R uN = ux * s.Nx + uy * s.Ny, iad = s.ia * s.id;
    const R nb = b * iad * tb;             // adjoint of u.N
    const R db = -s.t * s.id * tb;         // of d
    const R ab = -s.ia * s.ia * ng - s.t * s.ia * tb + db;  // of a
    const R bb = uN * iad * tb - s.uu * db;                 // of b
    C.ie += R(0.5) * bb;
    R uub = -b * db;                       // of |u|^2
    R epb = B.ep + k.a_ep * ab - (qxx + qyy);
    const R Nxb = s.ia * B.gx + nb * ux, Nyb = s.ia * B.gy + nb * uy;
    B.ux += s.t * B.gx + nb * s.Nx;
    B.uy += s.t * B.gy + nb * s.Ny;
    m.hx = Nxb;
    m.hy = Nyb;
    // N = c h + u (Q/2 sigma - T) + T F/2
    const R qT = k.hq_sigma - s.T, hT = R(0.5) * s.T;
    B.ux += qT * Nxb;
    B.uy += qT * Nyb;
    B.Fx += hT * Nxb;
    B.Fy += hT * Nyb;
    R thb = B.th + R(0.5) * (Fx * Nxb + Fy * Nyb) - (ux * Nxb + uy * Nyb);
    // ep = e1 sum f + e2 u.F + e3 |u|^2
    const R e2 = k.e2_ie * s.ie, e3 = k.e3_ie * s.ie;
    m.f0 = k.e1 * epb;
    m.fxx = qxx;
    m.fyy = qyy;
    const R uFb = e2 * epb;
    uub += e3 * epb;
    C.ie += epb * (k.e2_ie * (ux * Fx + uy * Fy) + k.e3_ie * s.uu);
    B.ux += uFb * Fx + R(2) * uub * ux;
    B.uy += uFb * Fy + R(2) * uub * uy;
    B.Fx += uFb * ux;
    B.Fy += uFb * uy;
    // F = e a - (a1 + a2 |u|) u
    const R dragb = -(B.Fx * ux + B.Fy * uy);
    B.ux -= s.drag * B.Fx;
    B.uy -= s.drag * B.Fy;
    C.e += k.ax * B.Fx + s.Gy * B.Fy;
    R Gyb = s.e * B.Fy;
    C.a1 += dragb;
    C.a2 += s.um * dragb;
    const R umb = s.a2 * dragb;
    // u = v/den, |u| = |v|/den, den = c0 + sqrt(c0^2 + c1 |v|), c0 = (1 + a1/2)/2, c1 = a2/2
    const R denb = -s.iden * (ux * B.ux + uy * B.uy + s.um * umb);
    const R rb = R(0.5) * denb * lrcp(s.rs);
    C.a1 += R(0.25) * (denb + R(2) * s.c0 * rb);
    C.a2 += R(0.5) * s.vm * rb;
    const R vmb = s.iden * umb + s.c1 * rb;
    // |v| is not differentiable at 0, but there it only enters times v: 0
    const R vs = s.vm > R(0) ? vmb * lrcp(s.vm) : R(0);
    const R vxb = s.iden * B.ux + vs * s.vx, vyb = s.iden * B.uy + vs * s.vy;
    m.fx = k.inv_rho0 * vxb;
    m.fy = k.inv_rho0 * vyb;
    C.e += R(0.5) * (k.ax * vxb + s.Gy * vyb);
    Gyb += R(0.5) * s.e * vyb;
    thb += k.gbeta * Gyb;
    m.h0 = k.inv_sigma * thb;
    return m;
}

// d e-total of a node's porosity from its constants' adjoints: 1/e, and with
// q = 1/e - 1, a1 = A1 q^2, a2 = A2 q/e (field_cell).
template <class R>
__device__ __forceinline__ R porosity_adjoint(const KConst<R>& k, R ie, const CellBar<R>& C) {
    const R q = ie - R(1), ie2 = ie * ie;
    return C.e - ie2 * (C.ie - R(2) * k.nnuK_q2 * q * C.a1 - k.nFK_q * (q + ie) * C.a2);
}

// T(x_ff) adjoints waiting at node (x, y): its thermal value along c_i is
// pulled by s = (x, y) + c_i, and the adiabatic wall nodes whose x_ff is s left
// theirs in Vff.
template <class R>
__device__ __forceinline__ R pending_ff(const KConst<R>& k, const R* __restrict__ Vff, int sx, int sy) {
    const bool wW = k.bc[SW] != BC_PERIODIC, wS = k.bc[SS] != BC_PERIODIC;
    if (!wW) sx = sx < 0 ? sx + k.nx : (sx >= k.nx ? sx - k.nx : sx);
    if (!wS) sy = sy < 0 ? sy + k.ny : (sy >= k.ny ? sy - k.ny : sy);
    const bool inx = wW ? sx >= 1 && sx <= k.nx - 2 : true, iny = wS ? sy >= 1 && sy <= k.ny - 2 : true;
    if (!inx || !iny) return R(0);
    R v = R(0);
    const bool W2 = k.bc[SW] == BC_ADIABATIC && sx == 2, E2 = k.bc[SE] == BC_ADIABATIC && sx == k.nx - 3;
    const bool S2 = k.bc[SS] == BC_ADIABATIC && sy == 2, N2 = k.bc[SN] == BC_ADIABATIC && sy == k.ny - 3;
    if (W2) v += Vff[at_of(k, 0, sy)];
    if (E2) v += Vff[at_of(k, k.nx - 1, sy)];
    if (S2) v += Vff[at_of(k, sx, 0)];
    if (N2) v += Vff[at_of(k, sx, k.ny - 1)];
    // a corner is adiabatic when both its walls are
    if (W2 && S2) v += Vff[at_of(k, 0, 0)];
    if (E2 && S2) v += Vff[at_of(k, k.nx - 1, 0)];
    if (W2 && N2) v += Vff[at_of(k, 0, k.ny - 1)];
    if (E2 && N2) v += Vff[at_of(k, k.nx - 1, k.ny - 1)];
    return v * k.inv_sigma;
}

// Adjoints of node (x, y)'s 17 post-collision values.
template <class R>
__device__ __forceinline__ void load_lambda(const KConst<R>& k, const R* __restrict__ lam, const R* __restrict__ Vff,
                                            bool ff, int x, int y, R* lf, R* lh) {
    const R* l = lam + at_of(k, x, y);
#pragma unroll
    for (int i = 1; i < 9; ++i) lf[i] = l[(long long)(i - 1) * k.plane];
#pragma unroll
    for (int i = 0; i < 9; ++i) lh[i] = l[(long long)(8 + i) * k.plane];
    lf[0] = R(0);
    // x_ff lies two nodes inside a wall: only nodes within three of one collect
    if (ff && (x <= 3 || y <= 3 || x >= k.nx - 4 || y >= k.ny - 4)) {
#pragma unroll
        for (int i = 0; i < 9; ++i) lh[i] += pending_ff(k, Vff, x + cx_of(i), y + cy_of(i));
    }
}

// Interior nodes (columns x0 .. x0 + nxi - 1, rows likewise), those beside a wall
// (the ring: S and N rows, then the W and E columns without them) and the
// others numbered apart; x, y hold x0, y0 on entry.
struct Interior {
    bool wx, wy;
    int nxi, nyi, rows, cols;  // rows, cols: without the ring
    template <class R>
    __host__ __device__ explicit Interior(const KConst<R>& k)
        : wx(k.bc[SW] != BC_PERIODIC), wy(k.bc[SS] != BC_PERIODIC), nxi(k.nx - (wx ? 2 : 0)), nyi(k.ny - (wy ? 2 : 0)),
          rows(nyi - (wy ? 2 : 0)), cols(nxi - (wx ? 2 : 0)) {}
    __host__ __device__ int ring() const { return (wy ? 2 * nxi : 0) + (wx ? 2 * rows : 0); }
    __host__ __device__ long long inner() const { return (long long)rows * cols; }
    __device__ __forceinline__ void ring_node(int n, int& x, int& y) const {
        if (wy) {
            if (n < nxi) { x += n; return; }
            n -= nxi;
            if (n < nxi) { x += n; y += nyi - 1; return; }
            n -= nxi;
        }
        y += (wy ? 1 : 0) + (n < rows ? n : n - rows);
        if (n >= rows) x += nxi - 1;
    }
    __device__ __forceinline__ void inner_node(long long n, int& x, int& y) const {
        const int r = (int)(n / cols);
        x += (wx ? 1 : 0) + (int)(n - (long long)r * cols);
        y += (wy ? 1 : 0) + r;
    }
};

// One adjoint step.  state: s_n; lam, Vff: adjoints of s_{n+1}; lam_prev,
// Vff_prev: those of s_n (places no interior node pulls are never written and
// stay 0).  ff: some wall is adiabatic.  early: the state was complete before
// the previous launch began, so it may be read before the grid dependency is
// resolved.
// The first ring_blocks blocks take the nodes beside a wall, 32 a block: their
// first warp the node's own collision, their second one those of the wall nodes
// it feeds, at the same time (in one thread the second chain follows the first,
// and every warp of a small lattice holds such a node); the first warp adds
// the two and goes on.  The other blocks take 64 nodes.
// Bound: 256^2 FP32 fits L2 and one wave of warps; the step takes about the
// latency of its chain (loads, ~600 dependent operations, stores).  Before, 9
// to 11 forward-mode passes a node in a thread each, then a combining and a
// gathering launch: whole calls with 256 steps at 256^2 FP32 took 38.0 ms
// against 7.0 ms, with 100 steps at 65 x 49 FP64 45.7 against 6.3 ms (lattice,
// uploads, forward and recomputed steps included; 7.5 and 8.4 ms with the wall nodes' chains in the
// threads of the nodes they hang on).
constexpr int kAdjNodes = 64, kAdjRing = 32;
template <class R> struct AdjLaunch { static constexpr int blocks = 8; };
template <> struct AdjLaunch<double> { static constexpr int blocks = 4; };

template <class R, class S, bool TAU1>
__global__ void __launch_bounds__(kAdjNodes, AdjLaunch<R>::blocks)
k_adj_step(const __grid_constant__ KConst<R> k, const S* __restrict__ state, const R* __restrict__ lam,
           const R* __restrict__ Vff, R* __restrict__ lam_prev, R* __restrict__ Vff_prev, double* __restrict__ g_eps,
           double* __restrict__ g_tb, int ring_blocks, bool ff, bool early) {
    constexpr int kShared = TAU1 ? 10 : 27;
    __shared__ R part[kShared][kAdjRing];  // what the wall nodes add, per node of the ring
    if (!early) asm volatile("griddepcontrol.wait;" ::: "memory");
    const Interior in(k);
    const bool ring = (int)blockIdx.x < ring_blocks;
    const bool walls = ring && threadIdx.x >= kAdjRing;  // this thread's role
    const int slot = threadIdx.x & (kAdjRing - 1);
    int x = in.wx ? 1 : 0, y = in.wy ? 1 : 0;
    bool live;
    if (ring) {
        const int n = (int)blockIdx.x * kAdjRing + slot;
        live = n < in.ring();
        if (live) in.ring_node(n, x, y);
    } else {
        const long long n = (long long)((int)blockIdx.x - ring_blocks) * kAdjNodes + threadIdx.x;
        live = n < in.inner();
        if (live) in.inner_node(n, x, y);
    }
    Pops<R> P;
    pull(k, state, x, y, P);
    const AdjState<R> s = adjoint_state(k, node_eps(k, x, y), row_ay(k, y), P.f, P.h);
    if (early) asm volatile("griddepcontrol.wait;" ::: "memory");
    // only now may the next step's blocks start: their early reads then come
    // after the launch before this one
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    StateBar<R> B = {};
    CellBar<R> C = {};
    R lf[9], lh[9], vf[9], vh[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) vf[i] = vh[i] = R(0);
    if (live && !walls) {
        load_lambda(k, lam, Vff, ff, x, y, lf, lh);
        emit_adjoint<true>(k, s.ie, TAU1 ? R(1) : R(1) - k.omf, TAU1 ? R(1) : R(1) - k.omT, s.ux, s.uy, s.Fx, s.Fy, s.ep,
                           s.T, s.gx, s.gy, lf, lh, B, C);
        if constexpr (!TAU1) {
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                vf[i] = k.omf * lf[i];
                vh[i] = k.omT * lh[i];
            }
        }
    }
    if (live && walls) {
        // the wall nodes whose x_f this node is
        const int bx = in.wx && x == 1 ? 0 : (in.wx && x == k.nx - 2 ? k.nx - 1 : -1);
        const int by = in.wy && y == 1 ? 0 : (in.wy && y == k.ny - 2 ? k.ny - 1 : -1);
#pragma unroll 1
        for (int m = 0; m < 3; ++m) {
            const int X = m == 1 ? x : bx, Y = m == 0 ? y : by;  // W/E side, S/N side, corner
            if (X < 0 || Y < 0) continue;
            const WallInfo w = classify(k, X, Y);
            load_lambda(k, lam, Vff, ff, X, Y, lf, lh);
            const R eb = k.eps_field ? k.eps_field[(long long)Y * k.nx + X] : k.eps;
            const Cell<R> cb = k.eps_field ? field_cell<R>(k, eb) : k.cell;
            R thb = R(0), thff = R(0);
            if (w.tside >= 0) {
                thb = k.T_bc[w.tside] - k.T0;
            } else {
                thff = (pull_hsum<R, R, S>(k, state, w.xff, w.yff) + R(0.5) * k.Q) * k.inv_sigma;
                thb = (R(4) * s.th - thff) * (R(1) / R(3));
            }
            const bool cutx = w.tside < 0 && w.fixgx, cuty = w.tside < 0 && w.fixgy;
            const R gx = cutx ? R(0) : s.gx, gy = cuty ? R(0) : s.gy;
            const R ux = k.u_bc[w.uside][0], uy = k.u_bc[w.uside][1], um = k.u_abs[w.uside];
            const R Gy = k.gbeta * thb + row_ay(k, Y), drag = -cb.nnuK - cb.nFK * um;
            const R Fx = cb.eps * k.ax - drag * ux, Fy = cb.eps * Gy - drag * uy;
            const R p = s.ep * s.ie, ep = k.eps_field ? p * cb.eps : s.ep;
            StateBar<R> D = {};
            CellBar<R> E = {};
            emit_adjoint<true>(k, cb.ie, R(1), R(1), ux, uy, Fx, Fy, ep, k.T0 + thb, gx, gy, lf, lh, D, E);
            // F = e a - (a1 + a2 |u_b|) u_b with u_b given
            const R dragb = -(D.Fx * ux + D.Fy * uy);
            E.a1 += dragb;
            E.a2 += um * dragb;
            E.e += k.ax * D.Fx + Gy * D.Fy;
            const R thbb = D.th + cb.eps * k.gbeta * D.Fy;
            if (w.tside >= 0) {
                g_tb[(long long)Y * k.nx + X] += double(thbb);
            } else {
                B.th += (R(4) / R(3)) * thbb;
                Vff_prev[at_of(k, X, Y)] = -(R(1) / R(3)) * thbb;
            }
            if (k.eps_field) {
                B.ep += D.ep * s.ie * cb.eps;
                C.ie += D.ep * s.ep * cb.eps;
                E.e += D.ep * p;
                g_eps[(long long)Y * k.nx + X] += double(porosity_adjoint(k, cb.ie, E));
            } else {
                B.ep += D.ep;
            }
            B.Sxx += D.Sxx;
            B.Syy += D.Syy;
            B.Sxy += D.Sxy;
            if (!cutx) B.gx += D.gx;
            if (!cuty) B.gy += D.gy;
            if constexpr (!TAU1) {
                // (1 - 1/tau)[f(x_f) - f^eq(x_f)]
                emit_adjoint<false>(k, s.ie, -k.omf, -k.omT, s.ux, s.uy, s.Fx, s.Fy, s.ep, s.T, s.gx, s.gy, lf, lh, B, C);
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    vf[i] += k.omf * lf[i];
                    vh[i] += k.omT * lh[i];
                }
            }
        }
        R* o = &part[0][slot];
        const R v[10] = {B.th, B.ep, B.Sxx, B.Syy, B.Sxy, B.gx, B.gy, C.ie, B.ux, B.uy};
#pragma unroll
        for (int q = 0; q < 10; ++q) o[q * kAdjRing] = v[q];
        if constexpr (!TAU1) {
#pragma unroll
            for (int i = 1; i < 9; ++i) o[(9 + i) * kAdjRing] = vf[i];
#pragma unroll
            for (int i = 0; i < 9; ++i) o[(18 + i) * kAdjRing] = vh[i];
        }
    }
    if (ring) {
        __syncthreads();
        if (walls) return;
        const R* o = &part[0][slot];
        R* b[10] = {&B.th, &B.ep, &B.Sxx, &B.Syy, &B.Sxy, &B.gx, &B.gy, &C.ie, &B.ux, &B.uy};
#pragma unroll
        for (int q = 0; q < 10; ++q) *b[q] += live ? o[q * kAdjRing] : R(0);
        if constexpr (!TAU1) {
#pragma unroll
            for (int i = 1; i < 9; ++i) vf[i] += live ? o[(9 + i) * kAdjRing] : R(0);
#pragma unroll
            for (int i = 0; i < 9; ++i) vh[i] += live ? o[(18 + i) * kAdjRing] : R(0);
        }
    }
    if (!live) return;
    const SumsBar<R> m = moments_adjoint(k, s, B, C);
    if (k.eps_field) g_eps[(long long)y * k.nx + x] += double(porosity_adjoint(k, s.ie, C));
    // pulled value i of this node came from (x, y) - c_i
    const int xm = x == 0 ? k.nx - 1 : x - 1, xp = x == k.nx - 1 ? 0 : x + 1;
    const int ym = y == 0 ? k.ny - 1 : y - 1, yp = y == k.ny - 1 ? 0 : y + 1;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int cx = cx_of(i), cy = cy_of(i);
        R* o = lam_prev + at_of(k, cx > 0 ? xm : (cx < 0 ? xp : x), cy > 0 ? ym : (cy < 0 ? yp : y));
        const R rx = R(cx), ry = R(cy);
        if (i > 0)
            o[(long long)(i - 1) * k.plane] = vf[i] + m.f0 + rx * m.fx + ry * m.fy + rx * rx * m.fxx + ry * ry * m.fyy + rx * ry * m.fxy;
        o[(long long)(8 + i) * k.plane] = vh[i] + m.h0 + rx * m.hx + ry * m.hy;
    }
}

// Seed: lambda_n(y, q) = dL/dT(s) / sigma for the thermal planes, where s is
// the interior node that pulls (y, q) (T = T0 + (sum h + Q/2)/sigma).
template <class R>
__global__ void k_adj_seed(const __grid_constant__ KConst<R> k, const double* __restrict__ dLdT, R* __restrict__ lam) {
    const int x = blockIdx.x * kAdjBlock + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= k.nx) return;
    const bool px = k.bc[SW] == BC_PERIODIC, py = k.bc[SS] == BC_PERIODIC;
    for (int q = 0; q < 17; ++q) {
        R v = R(0);
        if (q >= 8) {
            const int i = q - 8;
            int sx = x + cx_of(i), sy = y + cy_of(i);
            if (px) sx = (sx + k.nx) % k.nx;
            if (py) sy = (sy + k.ny) % k.ny;
            if (sx >= 0 && sx < k.nx && sy >= 0 && sy < k.ny && !classify(k, sx, sy).wall)
                v = R(dLdT[(long long)sy * k.nx + sx] * double(k.inv_sigma));
        }
        lam[q * k.plane + at_of(k, x, y)] = v;
    }
}

template <class R, class S>
cudaError_t launch_adj_step(const KConst<R>& k, const S* state, const R* lam, const R* Vff, R* lam_prev, R* Vff_prev,
                            double* g_eps, double* g_tb, bool early, cudaStream_t st) {
    const Interior in(k);
    const int ring_blocks = (in.ring() + kAdjRing - 1) / kAdjRing;
    const long long blocks = ring_blocks + (in.inner() + kAdjNodes - 1) / kAdjNodes;
    bool ff = false;
    for (int s = 0; s < 4; ++s) ff = ff || k.bc[s] == BC_ADIABATIC;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kAdjNodes);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (k.omf == R(0) && k.omT == R(0))
        return cudaLaunchKernelEx(&cfg, k_adj_step<R, S, true>, k, state, lam, Vff, lam_prev, Vff_prev, g_eps, g_tb, ring_blocks, ff, early);
    return cudaLaunchKernelEx(&cfg, k_adj_step<R, S, false>, k, state, lam, Vff, lam_prev, Vff_prev, g_eps, g_tb, ring_blocks, ff, early);
}

template <class R>
cudaError_t launch_adj_seed(const KConst<R>& k, const double* dLdT, R* lam, cudaStream_t st) {
    const dim3 grid((unsigned)((k.nx + kAdjBlock - 1) / kAdjBlock), (unsigned)k.ny);
    k_adj_seed<R><<<grid, kAdjBlock, 0, st>>>(k, dLdT, lam);
    return cudaGetLastError();
}

}  // namespace lbm

// ------------------------------------------------------------------- host

namespace {

// Host mirror of the wall classification (Sec. 3.4 readings).
struct HostWall {
    bool wall;
    int xs, ys, xff, yff, tside;
};

HostWall host_classify(const lbm_params& p, int x, int y) {
    HostWall w{};
    const bool onW = x == 0 && p.bc[0] != LBM_BC_PERIODIC;
    const bool onE = x == p.nx - 1 && p.bc[1] != LBM_BC_PERIODIC;
    const bool onS = y == 0 && p.bc[2] != LBM_BC_PERIODIC;
    const bool onN = y == p.ny - 1 && p.bc[3] != LBM_BC_PERIODIC;
    w.wall = onW || onE || onS || onN;
    const int dx = onW ? 1 : (onE ? -1 : 0), dy = onS ? 1 : (onN ? -1 : 0);
    w.xs = x + dx;
    w.ys = y + dy;
    w.xff = x + 2 * dx;
    w.yff = y + 2 * dy;
    const int xsd = onW ? 0 : (onE ? 1 : -1), ysd = onS ? 2 : (onN ? 3 : -1);
    w.tside = -1;
    if (xsd >= 0 && p.bc[xsd] == LBM_BC_DIRICHLET) w.tside = xsd;
    else if (ysd >= 0 && p.bc[ysd] == LBM_BC_DIRICHLET) w.tside = ysd;
    return w;
}

}  // namespace

namespace {

// lbm_adjoint keeps every state (segment = 0) while together they take no more.
constexpr size_t kKeepBytes = (size_t)256 << 20;

// Steps that one launch takes of the next `left`: two on FP32 lattices that have
// the two-step kernel.
template <class S>
int64_t steps_of_launch(const lbm_handle* h, int64_t left) {
    return std::is_same<S, float>::value && h->two_steps && left >= 2 ? 2 : 1;
}
// m = 1 or 2 steps from src to dst; with two, the state between them to mid
// (or nowhere, if null).
template <class R, class S>
cudaError_t launch_steps(const lbm_handle* h, const lbm::KConst<R>& k, int64_t m, const S* src, S* mid, S* dst,
                         int64_t step, cudaStream_t st) {
    if constexpr (std::is_same<S, float>::value)
        if (m == 2) return lbm::launch_two_steps(k, src, mid, dst, (uint32_t)(step / 2), h->sms, st);
    return lbm::launch_step(k, src, dst, (uint32_t)step, st);
}

template <class R, class S>
lbm_status run_adjoint(lbm_handle* h, const lbm::KConst<R>& k, int64_t n, int64_t seg_len, int side, double* loss,
                       double* dloss_deps, double* dloss_dTbc) {
    cudaStream_t st = h->stream;
    const lbm_params& p = h->prm;
    const size_t N = (size_t)p.nx * p.ny;
    const size_t sb = h->L.buf_bytes;  // one state
    // few and small states are all kept as the forward pass computes them, and
    // nothing is recomputed (65 x 49 FP64, 100 steps: 4.8 ms in this call
    // against 5.7 with checkpoints; the same in FP32 1.4 and 1.7); where the memory for that is not to be had,
    // checkpoints are
    bool keep = seg_len == 0 && (double)sb * (double)n <= (double)kKeepBytes;
    const int64_t seg = seg_len > 0 ? seg_len : (int64_t)ceil(sqrt((double)n));
    const size_t lam_bytes = 17 * (size_t)k.plane * sizeof(R);    // one adjoint state
    std::vector<void*> allocs;
    auto fail_free = [&](lbm_status s, const std::string& m) {
        for (void* a : allocs) cudaFreeAsync(a, st);
        cudaStreamSynchronize(st);
        return lbm_handle_fail(h, s, m);
    };
    auto alloc = [&](size_t bytes) -> void* {
        void* a = nullptr;
        if (cudaMallocAsync(&a, bytes, st) != cudaSuccess) return nullptr;
        allocs.push_back(a);
        return a;
    };
    R* lam0 = (R*)alloc(lam_bytes);
    R* lam1 = (R*)alloc(lam_bytes);
    const size_t ff_bytes = (size_t)k.plane * sizeof(R);
    R* ff0 = (R*)alloc(2 * ff_bytes);  // T(x_ff) adjoints left at the wall nodes, two buffers
    double* g = (double*)alloc(3 * N * sizeof(double));  // g_eps, g_tb, dL/dT
    char* segs = keep ? (char*)alloc(sb * (size_t)n) : nullptr;
    if (keep && !segs) {
        (void)cudaGetLastError();
        keep = false;
    }
    const int64_t K = keep ? n : seg, nseg = (n + K - 1) / K;
    char* ckpt = keep ? segs : (char*)alloc(sb * (size_t)nseg);
    if (!keep) segs = (char*)alloc(sb * (size_t)K);
    if (!ckpt || !segs || !lam0 || !lam1 || !ff0 || !g)
        return fail_free(LBM_ERR_OOM, "adjoint buffers (checkpoints grow as sqrt(n))");
    R* ff1 = ff0 + k.plane;
    double *g_eps = g, *g_tb = g + N, *dLdT = g + 2 * N;
    // lam1 holds 0 where no node ever writes (lam0 is written whole by the seed)
    if (cudaMemsetAsync(g, 0, 2 * N * sizeof(double), st) != cudaSuccess ||
        cudaMemsetAsync(lam1, 0, lam_bytes, st) != cudaSuccess || cudaMemsetAsync(ff0, 0, 2 * ff_bytes, st) != cudaSuccess)
        return fail_free(LBM_ERR_CUDA, "memset");

    // forward, keeping a checkpoint at the start of every segment
    const int64_t step0 = h->steps;
    auto kept = [&](int64_t t) { return (S*)(segs + sb * (size_t)t); };  // state t of the segment in hand
    for (int64_t t = 0; t < n;) {
        if (t % K == 0)
            if (cudaMemcpyAsync(ckpt + sb * (size_t)(t / K), h->buf(h->cur), sb, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
                return fail_free(LBM_ERR_CUDA, "checkpoint copy");
        // as many steps as one launch takes, up to the next checkpoint
        const int64_t m = steps_of_launch<S>(h, std::min(K - t % K, n - t));
        const bool last = t + m == n;  // the handle ends at step n
        cudaError_t e = keep ? launch_steps(h, k, m, (const S*)kept(t), m == 2 ? kept(t + 1) : (S*)nullptr,
                                            last ? (S*)h->buf(1 - h->cur) : kept(t + m), step0 + t, st)
                             : launch_steps(h, k, m, (const S*)h->buf(h->cur), (S*)nullptr, (S*)h->buf(1 - h->cur),
                                            step0 + t, st);
        if (e != cudaSuccess) return fail_free(LBM_ERR_CUDA, std::string("step kernel: ") + cudaGetErrorString(e));
        if (!keep || last) h->cur = 1 - h->cur;
        h->steps += m;
        ++h->launches;
        t += m;
    }
    // loss
    cudaError_t e = lbm::launch_nusselt(k, h->diag, (const S*)h->buf(h->cur), side, h->nu(), h->out(), st);
    if (e != cudaSuccess) return fail_free(LBM_ERR_CUDA, "nusselt kernels");
    if (cudaMemcpyAsync(loss, h->out(), sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return fail_free(LBM_ERR_CUDA, "loss copy");

    // seed: dL/dT per node, wall nodes resolved onto interior nodes
    std::vector<double> dT(N, 0.0);
    double dTbc[4] = {0, 0, 0, 0};
    const int nw = side <= 1 ? p.ny : p.nx;
    for (int j = 0; j < nw; ++j) {
        const double wj = (j == 0 || j == nw - 1) ? 0.5 : 1.0;
        const double sgn = (side == 0 || side == 2) ? 1.0 : -1.0;  // d_axis = sgn * d_inward
        const double base = -h->d.L / h->d.dT * sgn * wj / double(nw - 1);
        const double coef[3] = {-1.5 * base, 2.0 * base, -0.5 * base};
        for (int m = 0; m < 3; ++m) {
            int x, y;
            if (side == 0) { x = m; y = j; }
            else if (side == 1) { x = p.nx - 1 - m; y = j; }
            else if (side == 2) { x = j; y = m; }
            else { x = j; y = p.ny - 1 - m; }
            const HostWall w = host_classify(p, x, y);
            if (!w.wall) dT[(size_t)y * p.nx + x] += coef[m];
            else if (w.tside >= 0) dTbc[w.tside] += coef[m];
            else {
                dT[(size_t)w.ys * p.nx + w.xs] += coef[m] * 4.0 / 3.0;
                dT[(size_t)w.yff * p.nx + w.xff] -= coef[m] / 3.0;
            }
        }
    }
    if (cudaMemcpyAsync(dLdT, dT.data(), N * sizeof(double), cudaMemcpyHostToDevice, st) != cudaSuccess)
        return fail_free(LBM_ERR_CUDA, "seed copy");
    e = lbm::launch_adj_seed(k, dLdT, lam0, st);
    if (e != cudaSuccess) return fail_free(LBM_ERR_CUDA, "seed kernel");
    if (cudaStreamSynchronize(st) != cudaSuccess) return fail_free(LBM_ERR_CUDA, "seed");  // dT reused below

    // backward over the segments, recomputing each from its checkpoint
    R* lc = lam0;
    R* ln = lam1;
    for (int64_t sgi = nseg - 1; sgi >= 0; --sgi) {
        const int64_t t0 = sgi * K, len = std::min<int64_t>(K, n - t0);
        if (!keep && cudaMemcpyAsync(segs, ckpt + sb * (size_t)sgi, sb, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
            return fail_free(LBM_ERR_CUDA, "checkpoint restore");
        for (int64_t t = keep ? len : 1; t < len;) {
            const int64_t m = steps_of_launch<S>(h, len - t);
            e = launch_steps(h, k, m, (const S*)kept(t - 1), m == 2 ? kept(t) : (S*)nullptr, kept(t + m - 1), step0 + t0 + t - 1, st);
            if (e != cudaSuccess) return fail_free(LBM_ERR_CUDA, "recompute step");
            t += m;
        }
        for (int64_t t = len - 1; t >= 0; --t) {
            // the first launch after the recomputation waits before it reads the state
            e = lbm::launch_adj_step(k, (const S*)kept(t), lc, ff0, ln, ff1, g_eps, g_tb, keep || t < len - 1, st);
            if (e != cudaSuccess) return fail_free(LBM_ERR_CUDA, std::string("adjoint kernel: ") + cudaGetErrorString(e));
            std::swap(lc, ln);
            std::swap(ff0, ff1);
        }
    }
    // gradients
    std::vector<double> hg(N);
    if ((dloss_deps && cudaMemcpyAsync(dloss_deps, g_eps, N * sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess) ||
        cudaMemcpyAsync(hg.data(), g_tb, N * sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return fail_free(LBM_ERR_CUDA, "gradient copy");
    for (int y = 0; y < p.ny; ++y)
        for (int x = 0; x < p.nx; x += (y == 0 || y == p.ny - 1 || p.nx < 2) ? 1 : p.nx - 1) {
            const HostWall w = host_classify(p, x, y);
            if (w.wall && w.tside >= 0) dTbc[w.tside] += hg[(size_t)y * p.nx + x];
        }
    if (dloss_dTbc) memcpy(dloss_dTbc, dTbc, sizeof(dTbc));
    for (void* a : allocs) cudaFreeAsync(a, st);
    if (cudaStreamSynchronize(st) != cudaSuccess) return lbm_handle_fail(h, LBM_ERR_CUDA, "adjoint cleanup");
    return LBM_OK;
}

}  // namespace

extern "C" lbm_status lbm_adjoint(lbm_handle* h, int64_t n_steps, int64_t segment, int side, double* loss,
                                  double* dloss_deps, double* dloss_dTbc) {
    const lbm_host::NvtxRange range("lbm_adjoint");
    if (!h) return LBM_ERR_ARG;
    if (n_steps < 1 || segment < 0 || side < 0 || side > 3 || !loss)
        return lbm_handle_fail(h, LBM_ERR_ARG, "bad step count, segment, side or null loss");
    if (h->prm.precision == LBM_F16)
        return lbm_handle_fail(h, LBM_ERR_ARG, "the adjoint runs on FP64 or FP32 storage");
    if (h->moments_kind())
        return lbm_handle_fail(h, LBM_ERR_ARG, "the adjoint runs on population storage, not on a moment state");
    if (h->nonfinite) return lbm_handle_fail(h, LBM_ERR_NONFINITE, "non-finite velocity or temperature");
    const bool field = h->prm.precision == LBM_F64 ? h->k64.eps_field != nullptr : h->k32.eps_field != nullptr;
    if (dloss_deps && !field)
        return lbm_handle_fail(h, LBM_ERR_ARG, "a porosity gradient needs a porosity field (lbm_set_fields)");
    if ((side <= 1 ? h->prm.nx : h->prm.ny) < 3)
        return lbm_handle_fail(h, LBM_ERR_ARG, "the one-sided difference needs 3 nodes");
    if (h->prm.precision == LBM_F64)
        return run_adjoint<double, double>(h, h->k64, n_steps, segment, side, loss, dloss_deps, dloss_dTbc);
    return run_adjoint<float, float>(h, h->k32, n_steps, segment, side, loss, dloss_deps, dloss_dTbc);
}
