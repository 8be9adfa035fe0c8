// Arguments of the step kernels and the per-cell source arithmetic that the
// float (rt_step.cu) and double (rt_step64.cu) kernels share.
#pragma once

#include <cuda_runtime.h>

#include <cmath>

#include "rt_internal.cuh"
#include "rt_step_common.cuh"
#include "rt_step_tile.cuh"

namespace rt {
namespace step {

// The Lorentz factor in Gamma = gamma (1 -+ v.n / c) (Sec. 2.3) of a cell
// with v / c = (bx, by, bz): 1 for the first-order transformation, else
// (1 - v^2 / c^2)^(-1/2).
__device__ __forceinline__ float rsqrt_r(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rsqrt_r(double x) { return rsqrt(x); }
template <typename R> __device__ __forceinline__ R frame_gamma(int boost, R bx, R by, R bz) {
  return boost ? rsqrt_r(R(1) - fma(bx, bx, fma(by, by, bz * bz))) : R(1);
}

// Temperature quartic of one interior cell and its emission term
// q = dt cbar rho (kP B + kS J~).  With w~ normalised, x_a = dt cbar rho
// (kJ + kS) Gamma_a and the sums S_I, S_G of Eq. (Jcom), S_1 = sum w~ / (1 + x):
//   D = 1 - dt cbar rho kS S_G = S_1 + dt cbar rho kJ S_G,
//   1 - dt cbar rho kJ S_G / D = S_1 / D,
// so the quartic alpha T^4 + rho c_v T = g of Eq. (com rad thermal disc) has
// alpha = dt c a rho kP S_1 / D and g = (e - kinetic) + dt c 4 pi rho kJ S_I / D:
// sums of positive terms, no cancellation when x >> 1.  The weight
// normalisation cancels in every ratio.  Sets status bits in `bad`.
template <typename R>
__device__ __forceinline__ double source_q(const StepArgs<R> &a, const GasStatic &g,
                                           const GasDyn &d, double SI, double SG, double S1,
                                           unsigned &bad) {
  const double dJ = a.k_dcr * g.rkJ, dP = a.k_dcr * g.rkP, dS = a.k_dcr * g.rkS;
  const double rU = rcp(fma(dJ, SG, S1));
  const double kin = 0.5 * (d.mx * d.mx + d.my * d.my + d.mz * d.mz) * g.inv_rho;
  const double alpha = a.k_alpha * g.rkP * S1 * rU;
  const double eint = d.e - kin;
  const double gq = eint + a.k_g * g.rkJ * SI * rU;
  double T = 0.0, dPT = dP;  // dPT: dP with kappa_P at T^{n+1}
  if (!(gq >= 0.0) || !(alpha >= 0.0)) {
    bad |= ST_NONFINITE;
  } else if (a.beta_P == 0.0) {
    if (quartic_root(alpha, g.rcv, gq, quotient(eint, g.rcv), 1e-15, a.newton_max_iter, &T))
      bad |= ST_NONCONV;
  } else {
    // kappa_P (T/T_ref)^beta_P T^4 = kappa_P T_ref^-beta_P T^(4 + beta_P)
    if (power_root(alpha * a.tref_mbP, 4.0 + a.beta_P, g.rcv, gq, eint / g.rcv, 1e-15,
                   a.newton_max_iter, &T))
      bad |= ST_NONCONV;
    dPT = dP * pow(T / a.T_ref, a.beta_P);
  }
  const double B = a.a_rad * (T * T) * (T * T) * (1.0 / (4.0 * kPi));
  const double J = fma(dPT * B, SG, SI) * rU;  // the J~ of Eq. (Jcom)
  return fma(dPT, B, dS * J);
}

// The gas exchange of cell cl (Eqs. gas1, gas2) from its sums dE = sum w dI,
// d(xyz) = sum w n dI, dI = I* - I': e and m of an interior cell, the tally of a
// boundary or emitter cell; the frame velocity and internal energy of the next
// step; and the cell's status bits.  One lane per cell.
template <typename R, bool MOVING>
__device__ __forceinline__ void gas_exchange(const StepArgs<R> &a, int64_t cl, const GasStatic &gs,
                                             GasDyn d, R sE, R sx, R sy, R sz, unsigned bad) {
  // dE_gas = (c/cbar) 4 pi sum w dI, d(rho v) = (4 pi c sum w n dI) / (c cbar)
  const double dE = a.k_fe * (double)sE;
  const double dx = a.k_fm * (double)sx, dy = a.k_fm * (double)sy, dz = a.k_fm * (double)sz;
  if (!a.commit) {
    // stage 1 of the van Leer step: the gas update is discarded
  } else if (a.kind[cl] == RT_CELL_INTERIOR) {
    d.e += dE;
    d.mx += dx;
    d.my += dy;
    d.mz += dz;
    a.gd[cl] = d;
    // frame velocity and internal energy for the next step
    const double ir = gs.inv_rho;
    const double kin = 0.5 * (d.mx * d.mx + d.my * d.my + d.mz * d.mz) * ir;
    store4(a.cellv + 4 * cl, R(d.mx * ir), R(d.my * ir), R(d.mz * ir), R(d.e - kin));
    if (a.beta_J != 0.0) {
      // kappa_J of the next step, at its starting temperature
      const double rkJ = a.rkJ0[cl] * pow((d.e - kin) / gs.rcv / a.T_ref, a.beta_J);
      a.gs_w[cl].rkJ = rkJ;
      a.gs_w[cl].frkJ = (float)rkJ;
    }
  } else {
    double *x = a.ext + 4 * cl;
    x[0] += dE;
    x[1] += dx;
    x[2] += dy;
    x[3] += dz;
  }
  if (MOVING && a.gcl_rate && a.commit) {
    // the cell's volume for the next step, V^{n+1} = V^n + dt sum_f A w . n;
    // this step needed V^n >= dt max_a sum_f max(u, 0) (the float factor
    // carries a ~1e-6 relative error, inside the margin)
    const double V = a.volume[cl];
    if (a.dt * ((double)a.gcl_kv[cl] * a.gcl_kv_unit) > V * (1.0 + 1e-5)) bad |= ST_CFL;
    const double V1 = __dadd_rn(V, __dmul_rn(a.dt, a.gcl_rate[cl]));
    a.volume[cl] = V1;
    a.inv_vol_w[cl] = R(1.0 / V1);
  }
  if (bad) {
    atomicOr(a.status, bad);
    atomicMin(a.bad_cell, (unsigned long long)cl);
  }
}

// The kernel arguments of one step with explicit rows.
template <typename R> StepArgs<R> step_args(rt_state *s, double dt, const StepIO &io) {
  StepArgs<R> a;
  a.n_cells = s->n_cells;
  a.n_angles = s->n_angles;
  a.half = s->n_angles / 2;
  a.row = s->row_stride;
  a.ptr = s->d_ptr;
  a.nbr = s->d_nbr;
  a.slot = reinterpret_cast<const typename SlotOf<R>::type *>(s->d_slot);
  a.slot_nb = s->d_slot_nb;
  a.uface = s->d_uface;
  a.inv_vol = reinterpret_cast<const R *>(s->d_inv_vol);
  a.wface = s->d_wface;
  a.gs = s->d_gs;
  a.gd = s->d_gd;
  a.kind = s->d_kind;
  a.aux = s->d_aux;
  a.bc_row = s->d_bc_row;
  a.I0 = reinterpret_cast<const R *>(s->d_I0);
  a.ext = s->d_ext;
  a.dir = reinterpret_cast<const R *>(s->d_dir);
  a.wt2 = reinterpret_cast<const R *>(s->d_wt);
  a.I_in = reinterpret_cast<const R *>(io.in);
  a.I_out = reinterpret_cast<R *>(io.out);
  a.src_only = io.src_only ? 1 : 0;
  a.commit = io.commit ? 1 : 0;
  a.boost = s->params.boost;
  a.gcl_rate = s->d_gcl_rate;
  a.gcl_kv = s->d_gcl_kv;
  a.gcl_kv_unit = 1.0 / s->screen_scale;
  a.volume = s->d_volume;
  a.inv_vol_w = reinterpret_cast<R *>(s->d_inv_vol);
  a.beta_P = s->params.beta_P;
  a.beta_J = s->params.beta_J;
  a.T_ref = s->params.T_ref;
  a.tref_mbP = a.beta_P != 0.0 ? pow(a.T_ref, -a.beta_P) : 1.0;
  a.beta_P_f = (float)a.beta_P;
  a.T_ref_f = (float)a.T_ref;
  a.tref_mbP_f = (float)a.tref_mbP;
  a.rkJ0 = s->d_rkJ0;
  a.gs_w = s->d_gs;
  a.dt = dt;
  a.dt_r = R(dt);
  a.dt_cbar_r = R(dt * s->params.cbar);
  a.inv_c_r = R(1.0 / s->params.c);
  a.cellv = reinterpret_cast<R *>(s->d_cellv);
  a.cbar = s->params.cbar;
  a.c = s->params.c;
  a.a_rad = s->params.a_rad;
  a.rcv = s->params.r_gas / (s->params.gamma_gas - 1.0);
  a.k_dcr = dt * s->params.cbar;
  a.k_alpha = dt * s->params.c * s->params.a_rad;
  a.k_g = dt * s->params.c * 4.0 * kPi;
  a.k_fe = s->params.c / s->params.cbar * 4.0 * kPi;
  a.k_fm = 4.0 * kPi / s->params.cbar;
  a.newton_max_iter = s->params.newton_max_iter;
  // iterations held back for the float solve to go on from a change of 1e-4 to 1e-7
  constexpr int kSpare = 8;
  const bool quick = a.newton_max_iter >= 2 * kSpare;
  a.quick_iter = quick ? a.newton_max_iter - kSpare : a.newton_max_iter;
  a.quick_tol = quick ? 1e-4f : 1e-7f;
  a.float_quartic = s->params.float_quartic;
  a.k_dcr_f = (float)a.k_dcr;
  a.k_alpha_f = (float)a.k_alpha;
  a.k_g_f = (float)a.k_g;
  a.a_rad_4pi_f = (float)(s->params.a_rad / (4.0 * kPi));
  a.status = s->d_status;
  a.bad_cell = s->d_bad;
  a.kout = s->d_kout;
  a.w_uniform = s->w_uniform;
  a.w_uni = R(s->w_uni);
  return a;
}

}  // namespace step
}  // namespace rt
