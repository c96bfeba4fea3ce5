// lbm_step.cuh -- device code shared by the single-lattice and the batched
// step kernels (internal): block size, the store of one node and the
// out-of-line wall-node update.
#pragma once

#include "lbm_diag.cuh"

namespace lbm {

constexpr int kStepBlock = 128;
// Resident blocks per SM the step kernel is compiled for: 8 x 128 threads
// caps the FP32 kernel at 64 registers; the FP64 kernel keeps room to avoid
// spilling.
#ifndef LBM_F32_STEP_BLOCKS
#define LBM_F32_STEP_BLOCKS 8
#endif
template <class R> struct StepOccupancy { static constexpr int blocks = LBM_F32_STEP_BLOCKS; };
template <> struct StepOccupancy<double> { static constexpr int blocks = 3; };

template <class R, class S>
__device__ __forceinline__ void store_node(const KConst<R>& k, S* __restrict__ dst, long long at,
                                           const R* fo, const R* ho, Dither* dither = nullptr) {
    store_planes<S, R>(dst + at, k.plane, fo, ho, k.inv_scale, dither);
}

// PART 1: the flow planes alone, 2: the thermal planes alone (what only the
// others need is then not computed).
template <int PART, class R>
__device__ __forceinline__ void store_part(R* __restrict__ d, long long pl, const R* fo, const R* ho) {
    if constexpr (PART == 1) {
#pragma unroll
        for (int i = 1; i < 9; ++i) d[(i - 1) * pl] = fo[i];
    } else {
#pragma unroll
        for (int i = 0; i < 9; ++i) d[(8 + i) * pl] = ho[i];
    }
}

// Interior node of one step: the nine pull sources are 32-bit offsets from
// the node (periodic wrap by per-thread deltas), plane strides are uniform
// across the launch.  TAU1: tau_f = tau_T = 1 (FP16 storage then takes its
// scale in the collision weights).
template <class R, class S, bool EPS_FIELD, bool TAU1, int PART = 0>
__device__ __forceinline__ void interior_update(const KConst<R>& k, const S* __restrict__ src,
                                                S* __restrict__ dst, int x, int y, uint32_t step) {
    const int dxm = x == 0 ? k.nx - 1 : -1;
    const int dxp = x == k.nx - 1 ? 1 - k.nx : 1;
    const int dym = y == 0 ? (k.ny - 1) * k.pitch : -k.pitch;
    const int dyp = y == k.ny - 1 ? (1 - k.ny) * k.pitch : k.pitch;
    const int o[9] = {0, dxm, dym, dxp, dyp, dxm + dym, dxp + dym, dxp + dyp, dxm + dyp};
    const int pl = k.plane32;
    const int at = y * k.pitch + x;
    const S* __restrict__ c = src + at;
    const float sc = k.scale;
    R f[9], h[9];
#pragma unroll
    for (int i = 1; i < 9; ++i) f[i] = load_pop<S, R>(c + ((i - 1) * pl + o[i]), sc);
#pragma unroll
    for (int i = 0; i < 9; ++i) h[i] = load_pop<S, R>(c + ((8 + i) * pl + o[i]), sc);
    Cell<R> cell;
    if constexpr (EPS_FIELD) cell = field_cell<R>(k, k.eps_field[(long long)y * k.nx + x]);
    else cell = k.cell;
    R fo[9], ho[9];
    constexpr bool prescale = TAU1 && std::is_same<S, __half>::value;
    core_interior<TAU1>(k, cell, eps_ay(k, k, cell, y), f, h, fo, ho, prescale ? R(k.inv_scale) : R(1));
    if (PART != 1 && !lfinite(ho[0])) atomicOr(k.flag, 1);
    if constexpr (PART != 0) {
        store_part<PART>(dst + at, pl, fo, ho);
    } else {
        Dither dither((uint32_t)at, step);
        store_planes<S, R>(dst + at, pl, fo, ho, prescale ? 1.0f : k.inv_scale, &dither);
    }
}

// Wall node idx of a lattice in perimeter order: S row, N row, W column, E
// column (walled sides only; the columns skip the rows' corner nodes).
template <class R>
__device__ __forceinline__ void perimeter_node(const KConst<R>& k, int idx, int& x, int& y) {
    const bool wS = k.bc[SS] != BC_PERIODIC, wN = k.bc[SN] != BC_PERIODIC;
    const int nS = wS ? k.nx : 0, nN = wN ? k.nx : 0;
    const int y0 = wS ? 1 : 0, y1 = wN ? k.ny - 1 : k.ny;
    const int nW = k.bc[SW] != BC_PERIODIC ? y1 - y0 : 0;
    if (idx < nS) { x = idx; y = 0; return; }
    idx -= nS;
    if (idx < nN) { x = idx; y = k.ny - 1; return; }
    idx -= nN;
    if (idx < nW) { x = 0; y = y0 + idx; return; }
    idx -= nW;
    x = k.nx - 1;
    y = y0 + idx;
}

// Number of wall nodes in that order.
template <class R>
__host__ __device__ inline int perimeter_nodes(const KConst<R>& k) {
    const int wS = k.bc[SS] != BC_PERIODIC, wN = k.bc[SN] != BC_PERIODIC;
    const int inner = k.ny - wS - wN;
    return (wS + wN) * k.nx + ((k.bc[SW] != BC_PERIODIC) + (k.bc[SE] != BC_PERIODIC)) * inner;
}

// Where a wall node's update takes its pulled values from: the population
// buffer src in global memory.
template <class R, class S>
struct GlobalSource {
    const S* src;
    __device__ __forceinline__ void operator()(const KConst<R>& k, int x, int y, Pops<R>& P) const { pull(k, src, x, y, P); }
};

// Wall node (x, y) of one step.  At tau_f = tau_T = 1 the extrapolated
// non-equilibrium part vanishes and the node is the collision of its boundary
// state (core_boundary): one moment evaluation at x_f and one collision.
template <class R, class Source>
__device__ __forceinline__ void wall_node_tau1(const KConst<R>& k, const Source& source, int x, int y, R* fo, R* ho) {
    const WallInfo w = classify(k, x, y);
    Pops<R> P;
    source(k, w.xs, w.ys, P);
    R thff = R(0);
    if (w.tside < 0) {
        Pops<R> Q;
        source(k, w.xff, w.yff, Q);  // only h is used
        thff = core_theta(k, core_hsum(Q.h));
    }
    const Cell<R> cs = node_cell(k, w.xs, w.ys), cb = node_cell(k, x, y);
    CoreState<R> s = core_moments(k, cs, eps_ay(k, k, cs, w.ys), P.f, P.h);
    const Shear<R> S_ = core_shear(k, cs, s);
    const R thb = w.tside >= 0 ? k.T_bc[w.tside] - k.T0 : R(0);
    core_boundary(k, cs, cb, eps_ay(k, k, cb, y), k.u_bc[w.uside][0], k.u_bc[w.uside][1], k.u_abs[w.uside], w.tside >= 0,
                  w.fixgx != 0, w.fixgy != 0, thb, thff, s);
    if (k.u_abs[w.uside] == R(0)) {
        core_emit<true, true, true>(k, cb, s, lmul(k.f_ScS, S_.xx), lmul(k.f_ScS, S_.yy), lmul(k.f_ScS2, S_.xy), P.f,
                                    P.h, fo, ho, R(1));
    } else {
        R Qxx, Qyy, Q2;
        shear_form<true>(k, cb, s.ux, s.uy, s.Fx, s.Fy, S_, Qxx, Qyy, Q2);
        core_emit<true, true>(k, cb, s, Qxx, Qyy, Q2, P.f, P.h, fo, ho, R(1));
    }
    if (!lfinite(ho[0])) atomicOr(k.flag, 1);
}

// The same at other relaxation times, where the non-equilibrium part stays
// (wall_emit).  Every operation is spelled out here too: kernels that take one
// and two steps, from global and from shared memory, give the same bits.
template <class R, class Source>
__device__ __forceinline__ void wall_node_generic(const KConst<R>& k, const Source& source, int x, int y, R* fo, R* ho) {
    const WallInfo w = classify(k, x, y);
    Pops<R> P;
    source(k, w.xs, w.ys, P);
    R thff = R(0);
    if (w.tside < 0) {
        Pops<R> Q;
        source(k, w.xff, w.yff, Q);  // only h is used
        thff = core_theta(k, core_hsum(Q.h));
    }
    const Cell<R> cs = node_cell(k, w.xs, w.ys), cb = node_cell(k, x, y);
    const CoreState<R> s = core_moments(k, cs, eps_ay(k, k, cs, w.ys), P.f, P.h);
    const Shear<R> S_ = core_shear(k, cs, s);
    const R thb = w.tside >= 0 ? k.T_bc[w.tside] - k.T0 : R(0);
    CoreState<R> b = s;
    core_boundary(k, cs, cb, eps_ay(k, k, cb, y), k.u_bc[w.uside][0], k.u_bc[w.uside][1], k.u_abs[w.uside], w.tside >= 0,
                  w.fixgx != 0, w.fixgy != 0, thb, thff, b);
    wall_emit(k, cs, cb, s, S_, b, P.f, P.h, fo, ho);
    if (!lfinite(fo[1]) || !lfinite(ho[0])) atomicOr(k.flag, 1);
}

// Both out of line: only the 4(N - 1) wall threads take them.
template <class R, class S, int PART>
__device__ __noinline__ void wall_update_tau1(const KConst<R>& k, const S* __restrict__ src, S* __restrict__ dst,
                                              int x, int y, uint32_t step) {
    R fo[9], ho[9];
    wall_node_tau1(k, GlobalSource<R, S>{src}, x, y, fo, ho);
    if constexpr (PART != 0) {
        store_part<PART>(dst + (long long)y * k.pitch + x, k.plane, fo, ho);
    } else {
        Dither dither((uint32_t)(y * k.pitch + x), step);
        store_node(k, dst, (long long)y * k.pitch + x, fo, ho, &dither);
    }
}
template <class R, class S>
__device__ __noinline__ void wall_update_generic(const KConst<R>& k, const S* __restrict__ src, S* __restrict__ dst,
                                                 int x, int y, uint32_t step) {
    R fo[9], ho[9];
    wall_node_generic(k, GlobalSource<R, S>{src}, x, y, fo, ho);
    Dither dither((uint32_t)(y * k.pitch + x), step);
    store_node(k, dst, (long long)y * k.pitch + x, fo, ho, &dither);
}

template <class R, class S>
__device__ __forceinline__ void wall_update(const KConst<R>& k, const S* __restrict__ src, S* __restrict__ dst, int x,
                                            int y, uint32_t step) {
    if (k.omf == R(0) && k.omT == R(0)) wall_update_tau1<R, S, 0>(k, src, dst, x, y, step);
    else wall_update_generic(k, src, dst, x, y, step);
}

}  // namespace lbm
