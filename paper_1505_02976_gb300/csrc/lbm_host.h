// lbm_host.h -- host-side helpers shared by the C ABI entry points:
// parameter derivation and checks, workspace layout, kernel constants.
#pragma once

#include <cuda_fp16.h>
#include <math.h>
#include <string.h>

#include <string>

#include <nvtx3/nvToolsExt.h>

#include "../../include/lbm.h"
#include "lbm_internal.h"

namespace lbm_host {

constexpr double kCs2 = 1.0 / 3.0;
constexpr double kW0 = 4.0 / 9.0;
constexpr int NPLANES_HOST = lbm::NPLANES;

struct Derived {
    double L, T0, dT, U, gbeta, nu, nu_e, alpha_e, A, B, K, Feps, Q;
};

inline bool isnan_(double v) { return v != v; }

// Lattice constants from the problem statement (Sec. 2, Sec. 4, Eq. EQA&B,
// Eq. Therdiff, Appendix A): see the table in include/lbm.h.
inline lbm_status derive(const lbm_params* p, Derived* d, std::string* why) {
    d->L = isnan_(p->L) ? double(p->nx - 1) : p->L;
    d->T0 = isnan_(p->T0) ? 0.5 * (p->Th + p->Tc) : p->T0;
    d->dT = p->Th - p->Tc;
    d->U = p->Ma * sqrt(kCs2);
    d->gbeta = isnan_(p->gbeta) ? d->U * d->U / (d->dT * d->L) : p->gbeta;
    if (!isnan_(p->nu)) d->nu = p->nu;
    else if (!isnan_(p->A)) d->nu = kCs2 * (p->tau_f - p->A - 0.5) / p->J;
    else d->nu = d->U * d->L * sqrt(p->Pr / p->Ra);
    d->nu_e = p->J * d->nu;
    if (!isnan_(p->alpha_e)) d->alpha_e = p->alpha_e;
    else if (!isnan_(p->B)) d->alpha_e = p->sigma * kCs2 * (p->tau_T - p->B - 0.5);
    else d->alpha_e = d->nu / p->Pr;
    d->A = isnan_(p->A) ? p->tau_f - 0.5 - d->nu_e / kCs2 : p->A;
    d->B = isnan_(p->B) ? p->tau_T - 0.5 - d->alpha_e / (p->sigma * kCs2) : p->B;
    d->K = p->da_infinite ? INFINITY : (isnan_(p->K) ? p->Da * d->L * d->L : p->K);
    d->Feps = p->forchheimer ? 1.75 / sqrt(150.0 * p->eps * p->eps * p->eps) : 0.0;
    d->Q = isnan_(p->Q) ? p->Ra_I * d->alpha_e * d->dT / (p->Ra * d->L * d->L) : p->Q;
    auto bad = [&](const char* m) {
        if (why) *why = m;
        return LBM_ERR_PARAM_RANGE;
    };
    if (!(p->eps > 0.0 && p->eps <= 1.0)) return bad("porosity eps must lie in (0, 1]");
    if (!(p->tau_f > 0.5 && p->tau_T > 0.5)) return bad("relaxation times must exceed 1/2");
    if (!(d->A < p->tau_f - 0.5)) return bad("A must be below tau_f - 1/2 (positive viscosity)");
    if (!(d->B < p->tau_T - 0.5)) return bad("B must be below tau_T - 1/2 (positive diffusivity)");
    if (!(p->sigma > 0.0 && p->rho0 > 0.0)) return bad("sigma and rho0 must be positive");
    if (!(isfinite(d->gbeta) && isfinite(d->nu) && isfinite(d->alpha_e) && isfinite(d->T0) &&
          isfinite(d->Q)))
        return bad("derived constants are not finite (check Ra, Ra_I, Pr, Ma, Th - Tc)");
    return LBM_OK;
}

inline lbm_status check_shape(const lbm_params* p, std::string* why) {
    for (int s = 0; s < 4; ++s)
        if (p->bc[s] < 0 || p->bc[s] > 2) { *why = "unknown boundary kind"; return LBM_ERR_ARG; }
    if ((p->bc[0] == LBM_BC_PERIODIC) != (p->bc[1] == LBM_BC_PERIODIC) ||
        (p->bc[2] == LBM_BC_PERIODIC) != (p->bc[3] == LBM_BC_PERIODIC)) {
        *why = "a periodic side needs a periodic opposite side";
        return LBM_ERR_ARG;
    }
    if (p->nx < 1 || p->ny < 1 || p->ny > 65535 || p->nx > (1 << 24)) {
        *why = "lattice size out of range (1 <= nx, 1 <= ny <= 65535)";
        return LBM_ERR_ARG;
    }
    if ((p->bc[0] != LBM_BC_PERIODIC && p->nx < 4) || (p->bc[2] != LBM_BC_PERIODIC && p->ny < 4)) {
        *why = "a walled direction needs at least 4 nodes";
        return LBM_ERR_ARG;
    }
    if ((double)NPLANES_HOST * (double)((size_t)p->nx + 128) * (double)p->ny >= 2147483647.0) {
        *why = "lattice too large for 32-bit plane offsets (17 nx ny < 2^31)";
        return LBM_ERR_ARG;
    }
    if (p->precision < LBM_F64 || p->precision > LBM_F16 || p->moment_state < 0 || p->moment_state > 1) {
        *why = "unknown precision or state kind";
        return LBM_ERR_ARG;
    }
    if (p->moment_state && !(p->tau_f == 1.0 && p->tau_T == 1.0 && p->precision != LBM_F16)) {
        *why = "moment storage needs tau_f = tau_T = 1 and FP32 or FP64";
        return LBM_ERR_ARG;
    }
    return LBM_OK;
}

inline size_t elem_size(int precision) {
    return precision == LBM_F64 ? 8 : (precision == LBM_F32 ? 4 : 2);
}

inline size_t align256(size_t v) { return (v + 255) & ~size_t(255); }

// Host memory that CUDA knows nothing of (not page-locked, not managed).
inline bool pageable(const void* p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) == cudaSuccess) return a.type == cudaMemoryTypeUnregistered;
    (void)cudaGetLastError();
    return false;
}

// The four moment fields from the device area F (nx ny doubles each, one after
// the other) to outs (null: not wanted).  Pageable host fields that lie one
// after the other go in one copy: each costs 10 us before its first byte (256^2:
// 60 -> 35 us a call).  Other memory is copied field by field: fields that touch
// may belong to two allocations or registrations, which one copy must not span.
inline cudaError_t copy_moments(double* const outs[4], const double* F, size_t N, cudaMemcpyKind kind, cudaStream_t st) {
    bool joins[4];
    for (int q = 0; q < 4; ++q) joins[q] = outs[q] && kind == cudaMemcpyDeviceToHost && pageable(outs[q]);
    for (int q = 0; q < 4;) {
        int n = 1;
        while (joins[q] && q + n < 4 && joins[q + n] && outs[q + n] == outs[q] + n * N) ++n;
        if (outs[q]) {
            const cudaError_t e = cudaMemcpyAsync(outs[q], F + q * N, n * N * sizeof(double), kind, st);
            if (e != cudaSuccess) return e;
        }
        q += n;
    }
    return cudaSuccess;
}

// NVTX range over one entry point (visible to Nsight tools; a no-op
// otherwise).
struct NvtxRange {
    explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange&) = delete;
    NvtxRange& operator=(const NvtxRange&) = delete;
};

// Guard words: kGuardBytes of kGuardByte after every region of a workspace,
// written at creation and compared on request (lbm_check_guards), so that a
// kernel writing past the end of any region is detected.
constexpr size_t kGuardBytes = 256;
constexpr unsigned char kGuardByte = 0xA5;
constexpr int kMaxGuards = 32;

struct Layout {
    int pitch;
    size_t plane_elems, buf_bytes;
    size_t off_buf[2], off_fields, off_snap, off_nu, off_partial, off_eps, off_ay, off_out, off_flag, total;
    size_t off_mom[2], mom_bytes;  // moment state: two 9-plane buffers; off_buf[0] = off_buf[1] = expansion
    size_t guard[kMaxGuards];      // offsets of the guard words
    int n_guards;
};

inline Layout layout(const lbm_params* p) {
    Layout L;
    const size_t es = elem_size(p->precision);
    const size_t row = ((size_t)p->nx * es + 127) / 128 * 128;  // 128-byte rows
    L.pitch = int(row / es);
    L.plane_elems = (size_t)L.pitch * p->ny;
    L.buf_bytes = align256(L.plane_elems * es * lbm::NPLANES);
    const size_t N = (size_t)p->nx * p->ny;
    size_t o = 0;
    L.n_guards = 0;
    // each region is followed by a guard word
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o += align256(bytes);
        L.guard[L.n_guards++] = o;
        o += kGuardBytes;
        return at;
    };
    L.off_buf[0] = take(L.buf_bytes);
    if (p->moment_state) {
        L.off_buf[1] = L.off_buf[0];
        L.mom_bytes = align256(L.plane_elems * es * lbm::kMPlanes);
        L.off_mom[0] = take(L.mom_bytes);
        L.off_mom[1] = take(L.mom_bytes);
    } else {
        L.off_buf[1] = take(L.buf_bytes);
        L.mom_bytes = 0;
        L.off_mom[0] = L.off_mom[1] = 0;
    }
    // four fields; a lattice of one node needs a fifth value for the stream function
    L.off_fields = take((N == 1 ? 5 : 4 * N) * sizeof(double));
    L.off_snap = take(3 * N * sizeof(double));
    L.off_nu = take((size_t)(p->nx > p->ny ? p->nx : p->ny) * sizeof(double));
    L.off_partial = take((size_t)lbm::residual_blocks(p->nx, p->ny) * 4 * sizeof(double));
    L.off_eps = take(N * sizeof(double));
    L.off_ay = take((size_t)p->ny * sizeof(double));
    L.off_out = take(256);
    L.off_flag = take(256);
    L.total = o;
    return L;
}

template <class R>
inline lbm::KConst<R> make_kconst(const lbm_params* p, const Derived& d, const Layout& L, int* flag) {
    lbm::KConst<R> k;
    memset(&k, 0, sizeof(k));
    k.nx = p->nx;
    k.ny = p->ny;
    k.pitch = L.pitch;
    for (int s = 0; s < 4; ++s) k.bc[s] = p->bc[s];
    k.plane = (long long)L.plane_elems;
    const double eps = p->eps;
    const double nuK = isinf(d.K) ? 0.0 : d.nu / d.K;
    const double FK = isinf(d.K) ? 0.0 : d.Feps / sqrt(d.K);
    const double c0 = 0.5 * (1.0 + eps * 0.5 * nuK);
    const double c1 = eps * 0.5 * FK;
    k.rho0 = R(p->rho0);
    k.eps = R(eps);
    k.inv_eps = R(1.0 / eps);
    k.sigma = R(p->sigma);
    k.inv_sigma = R(1.0 / p->sigma);
    k.omf = R(1.0 - 1.0 / p->tau_f);
    // complementary to 1/tau_T as rounded to R: their sum multiplies the
    // temperature in each step
    k.omT = R(1) - R(1.0 / p->tau_T);
    k.tau_f = R(p->tau_f);
    k.kf = R(1.0 - 0.5 / p->tau_f);
    k.kT = R(1.0 - 0.5 / p->tau_T);
    k.A = R(d.A);
    k.B = R(d.B);
    k.T0 = R(d.T0);
    k.gbeta = R(d.gbeta);
    k.ax = R(p->ax);
    k.ay = R(p->ay);
    k.Q = R(d.Q);
    k.e_nuK = R(eps * nuK);
    k.e_FK = R(eps * FK);
    k.c0 = R(c0);
    k.c0sq = R(c0 * c0);
    k.c1 = R(c1);
    k.p_pref = R(kCs2 / (eps * (1.0 - kW0)));
    k.invD = R(1.0 / (kCs2 * p->rho0 * (d.A - p->tau_f)));
    k.a_const = R(kCs2 * p->sigma * (d.B - p->tau_T));
    k.bcoef = R(0.5 * (1.0 / eps - 1.0 / p->sigma));
    k.sT0 = R(p->sigma * d.T0);
    for (int s = 0; s < 4; ++s) {
        k.T_bc[s] = R(p->T_bc[s]);
        k.u_bc[s][0] = R(p->u_bc[s][0]);
        k.u_bc[s][1] = R(p->u_bc[s][1]);
    }
    k.scale = p->precision == LBM_F16 ? ldexpf(1.0f, -10) : 1.0f;
    k.inv_scale = 1.0f / k.scale;
    k.flag = flag;
    k.plane32 = (int)L.plane_elems;
    // the node update (lbm_core.cuh)
    const double rho0 = p->rho0, ie = 1.0 / eps, itf = 1.0 / p->tau_f, itT = 1.0 / p->tau_T;
    const double kf = 1.0 - 0.5 / p->tau_f, kT = 1.0 - 0.5 / p->tau_T;
    const double invD = 1.0 / (kCs2 * rho0 * (d.A - p->tau_f));
    // eps p = e1 sum f, e1 = c_s^2/(1 - w_0) = 3/5.  Each step multiplies the
    // pressure by 1 - 1/tau + e1 (3/tau) (4 w_1 + 4 w_5) = 1, so e1 is fitted
    // to the other factors as R holds them and its own rounding kept apart
    // (e1_lo): an error of one unit in the last place would build up.
    const R fA = R(3.0 * itf);
    const double wsum = 4.0 * (double(R(1) / R(9)) + double(lbm::w_diag<R>()));
    const double e1 = sizeof(R) == 4 ? (1.0 - double(k.omf)) / (double(fA) * wsum) : kCs2 / (1.0 - kW0);
    const double aS = 1.5 * itf * rho0 * d.A * invD;
    const double b0 = -0.5 / p->sigma, bc = 0.5 * ie + b0;
    k.inv_rho0 = R(1.0 / rho0);
    k.hq_sigma = R(0.5 * d.Q / p->sigma);
    k.half_Q = R(0.5 * d.Q);
    k.eay = R(eps * p->ay);
    k.half_ax = R(0.5 * p->ax);
    k.e1 = R(e1);
    k.e1_lo = R(e1 - double(k.e1));
    k.aS = R(aS);
    k.qu_ie = R(rho0 * (4.5 * itf - aS));
    k.qF_ie = R(rho0 * (9.0 * kf + aS));
    k.f_cu = R(3.0 * rho0 * itf);
    // In FP32 each step scales the momentum by 1 - 1/tau + (f_cu/rho0) (2 w_1 + 4
    // w_5) = 1 - 1.5e-8/tau.  In a clear fluid (Darcy drag smaller than that)
    // nothing else damps it, and tied roundings of f_cu u_x add to it: there the
    // drag coefficient gives it back (u of clear 90^2 to 400 x 301 cavities after
    // 100 steps against 64 bits: 2e-6 too small without, 3e-7 off with).  Where
    // there is drag it stays: there the roundings of c_0 and of the quotient in u
    // act on the momentum as much, with either sign (a gain fitted at any drag
    // measured 0.5 to 2.3 times the error of u).
    const double back = itf / kf * (1.0 - 3.0 * (2.0 * double(R(1) / R(9)) + 4.0 * double(lbm::w_diag<R>())));
    k.nnuK_0 = sizeof(R) == 4 && eps * nuK < back ? R(back) : R(0);
    // The sum of the collided f_1..f_8 is fA wsum (eps p) + tsum tr Q, and the
    // u u and u F parts of the two cancel (e2 = -(4/5) rho0 kf tau/eps, e3 =
    // -(2/5) rho0/eps): fitted to the factors as R holds them, since the rest
    // is a source of mass in each step.
    const double tsum = sizeof(R) == 4 ? 2.0 * double(R(1) / R(9)) + 4.0 * double(lbm::w_diag<R>()) + double(R(-1) / R(3)) * wsum : 4.0 / 27.0;
    const double c3 = sizeof(R) == 4 ? -tsum / (double(fA) * wsum) : -(4.0 / 27.0) / (3.0 * itf * (1.0 - kW0));
    k.e2_ie = R(c3 * (double(k.qF_ie) - double(k.aS) * rho0));
    k.e3_ie = R(c3 * (double(k.qu_ie) + double(k.aS) * rho0));
    k.cu2_ie = R(4.5 * itf * rho0);
    k.cuF_ie = R(9.0 * rho0 * kf);
    k.b_0 = R(b0);
    k.ug_b = R(6.0 * kT);
    k.kc_ie = R(4.5 * itT);
    k.a_ep = R(-0.5 / rho0);
    k.aS2 = R(2.0 * aS);
    k.f_ScS = R(1.5 * itf * rho0 * d.A);
    k.f_ScS2 = R(3.0 * itf * rho0 * d.A);
    k.fA_ep = fA;
    k.f_cF = R(3.0 * rho0 * kf);
    k.h_sig = R(itT * p->sigma);
    k.h_kQ = R(kT * d.Q);
    k.h_pT = R(itT * 3.0 / rho0);
    k.h0_pT = R(-itT * (5.0 / 3.0) / rho0);
    k.h_u3 = R(3.0 * itT);
    k.h_uQ = R(3.0 * kT * d.Q / p->sigma);
    k.h_g = R(itT * p->sigma * d.B);
    k.h_W = R(3.0 * kT);
    k.h_Wr = R(3.0 * kT / rho0);
    for (int s = 0; s < 4; ++s) k.u_abs[s] = R(sqrt(p->u_bc[s][0] * p->u_bc[s][0] + p->u_bc[s][1] * p->u_bc[s][1]));
    lbm::Cell<R>& c = k.cell;
    c.eps = R(eps);
    c.ie = R(ie);
    c.elo = R(1.0 / double(c.ie) - double(c.eps));
    c.eg = R(eps * d.gbeta);
    c.eax = R(eps * p->ax);
    c.heax = R(0.5 * eps * p->ax);
    c.c0 = R(c0);
    c.c0sq = R(c0 * c0);
    c.c1 = R(c1);
    c.nnuK = R(-eps * nuK + double(k.nnuK_0));
    c.nFK = R(-eps * FK);
    c.re = R(rho0 * ie);
    c.qu = R(rho0 * (4.5 * itf - aS) * ie);
    c.qF = R(rho0 * (9.0 * kf + aS) * ie);
    c.e2 = R(c3 * (double(c.qF) - double(k.aS) * rho0 * ie));
    // e3's own rounding would be the larger rest: kept apart (one operation a
    // node, 0.5 % of a 2048^2 case; without it p after 100 steps is 1.9 of 1.1e-6
    // off)
    const double e3 = c3 * (double(c.qu) + double(k.aS) * rho0 * ie);
    c.e3 = R(e3);
    c.e3_lo = R(e3 - double(c.e3));
    // the same term where S is given (walls, moment state): from q_u as rounded,
    // or e3 would not cancel its mass (p of the moment state at 2048^2
    // after 100 steps against 64 bits: 1.9e-6 off, so 1.1e-6)
    c.cu2 = R(double(c.qu) + double(k.aS) * rho0 * ie);
    c.cuF = R(9.0 * rho0 * kf * ie);
    c.b = R(bc);
    c.nb = R(-bc);
    c.ug = R(6.0 * kT * bc);
    c.kc = R(4.5 * itT * ie);
    // porosity field support (the field pointer is set by lbm_set_fields)
    k.eps_field = nullptr;
    k.kc_inv_ref = R(eps < 1.0 ? (1.0 - eps) * (1.0 - eps) / (eps * eps * eps) : 0.0);
    k.nu_over_Kref = R(nuK);
    k.inv_sqrt_Kref = R(isinf(d.K) ? 0.0 : 1.0 / sqrt(d.K));
    k.p_pref_eps = R(kCs2 / (1.0 - kW0));
    k.da_inf = p->da_infinite ? 1 : 0;
    // with q = (1 - e)/e: eps nu/K(e) = nu/K_ref q^2 / kc, eps F_eps/sqrt(K(e))
    // = 1.75/sqrt(150 kc K_ref) q/e, kc = (1 - eps)^2/eps^3 at the reference
    const double kc = eps < 1.0 ? (1.0 - eps) * (1.0 - eps) / (eps * eps * eps) : 0.0;
    const bool drag = !p->da_infinite && kc > 0.0 && !isinf(d.K);
    k.nnuK_q2 = R(drag ? -nuK / kc : 0.0);
    k.nFK_q = R(drag && p->forchheimer ? -1.75 / sqrt(150.0 * kc * d.K) : 0.0);
    k.forch = p->forchheimer ? 1 : 0;
    k.ay_row = nullptr;
    return k;
}


}  // namespace lbm_host
