// The temperature equation of a float state's cell (Eq. com rad thermal disc) and
// its emission term q, shared by the float step kernels.
#pragma once

#include <cuda_runtime.h>

#include "rt_internal.cuh"
#include "rt_step_args.cuh"

namespace rt {
namespace step {

// (float) of refine_root's result for the quartic alpha T^4 + beta T = g without
// FP64 instructions (GB300 issues a warp's over 64 cycles), so that every lane
// of the cell runs it and no block barrier is needed.  T0: the float root; bh =
// (float)beta.  One Newton step with the residual in pairs of floats
// (error-free products by FMA and two-sum, Dekker and Knuth).  Error of the
// result before its rounding, relative: residual 10 x 2^-48, f' 4 ulp of a step
// of at most 3e-7, the step's own quadratic error 1.5 (3e-7)^2, together below
// 2^-41; refine_root's (double residual, the same float f' and quotient) is
// smaller.  So where the unrounded result is farther than 2^-40 from the
// midpoint of two floats, both round to the same float.  Returns false where it
// is nearer (2^-16 of all cells), the step is larger, or an error term could
// underflow (each loses 2^-149 at most, so 2^-51 of g >= 2^-98; beta >= 2^-100 so that its
// low part loses 2^-49 of it): the caller then takes refine_root.  The limits lie below
// the thinnest gas in CGS units (rho c_v of 1e-30 g / cm^3 is 1e-22).  It matters: where
// every cell is past them a step takes 60 us instead of 52 (48^3 cells x 48 angles).
__device__ __forceinline__ bool refine_quartic(float alpha, double beta, float bh, float g,
                                               float T0, float *T) {
  const float p = T0 * T0, pe = fmaf(T0, T0, -p);
  const unsigned bhi = (unsigned)__double2hiint(beta), blo = (unsigned)__double2loint(beta);
  const int ex = (int)(bhi >> 20);  // biased; beta > 0
  // hot thin gas: the equation times 2^60, because what alpha T^2 loses below 2^-149 is
  // multiplied by T^2
  const float sc = g < p * 0x1p-99f ? 0x1p60f : 1.0f;
  const bool ok = p >= 0x1p-80f && p <= 0x1p80f && g >= 0x1p-98f && g <= 0x1p100f &&
                  g * sc >= p * 0x1p-100f && ex >= 923 && ex <= 1120;
  // beta - bh, by integers: the 29 mantissa bits below float's, less 2^29 if
  // bh was rounded up, scaled by 2^(exponent - 52) (in two factors: 2^-32 keeps the
  // first one a normal float for small beta)
  const unsigned trunc = ((unsigned)(ex - 896) << 23) | ((bhi & 0xfffffu) << 3) | (blo >> 29);
  const int up = __float_as_int(bh) - (int)trunc;  // 0 or 1
  const float bl = (float)((int)(blo & 0x1fffffffu) - (up << 29)) *
                   __int_as_float((ex - 1075 + 32 + 127) << 23) * (sc * 0x1p-32f);
  alpha *= sc;
  bh *= sc;
  g *= sc;
  const float r1 = alpha * p, r1e = fmaf(alpha, p, -r1) + alpha * pe;  // alpha T^2
  const float r = r1 * p;                                              // alpha T^4
  const float re = fmaf(r1, p, -r) + fmaf(r1, pe, r1e * p);
  const float s = bh * T0, se = fmaf(bh, T0, -s) + bl * T0;  // beta T
  const float t = r + s, tv = t - r;
  const float te = (r - (t - tv)) + (s - tv);
  const float f = (t - g) + ((te + re) + se);
  const float d = f * rcp(fmaf(4.0f * r1, T0, bh));
  const float Tr = T0 - d;
  *T = Tr;
  const float e = (T0 - Tr) - d;  // the unrounded result minus Tr
  const unsigned b = __float_as_uint(Tr);
  // half the distance to the next float on e's side (below a power of two half of that
  // above it)
  const unsigned lower = (b & 0x007fffffu) == 0 && e < 0.0f ? 25u : 24u;
  const float half = __uint_as_float((b & 0x7f800000u) - (lower << 23));
  return (ok && fabsf(fabsf(e) - half) > Tr * 0x1p-40f && fabsf(d) <= 3e-7f * Tr) ||
         (g == 0.0f && T0 == 0.0f);  // a dark vacuum: T = 0 exactly
}

// The temperature equation of a float state's cell in float: the
// coefficients of source_q from the float copies of the cell's opacities and
// the float angular sums (alpha multiplies T^(4 + beta_P) T_ref^-beta_P),
// with rU = 1 / D and dP, dS = dt cbar rho kappa_P, kappa_s.
struct QuarticF {
  float alpha, gq, rU, dP, dS;
};
__device__ __forceinline__ QuarticF float_coeffs(const StepArgs<float> &a, float rkP, float rkJ,
                                                 float rkS, float eint, float SI, float SG,
                                                 float S1) {
  QuarticF k;
  const float dJ = a.k_dcr_f * rkJ;
  k.dP = a.k_dcr_f * rkP;
  k.dS = a.k_dcr_f * rkS;
  k.rU = rcp(fmaf(dJ, SG, S1));
  k.alpha = a.k_alpha_f * rkP * S1 * k.rU;
  k.gq = eint + a.k_g_f * rkJ * SI * k.rU;
  if (a.beta_P_f != 0.0f) k.alpha *= a.tref_mbP_f;
  return k;
}
// Float root of the cell's equation from the pre-step temperature (returns
// 1 if Newton did not converge).
__device__ __forceinline__ int float_root(const StepArgs<float> &a, const QuarticF &k, float rcv,
                                          float eint, float *T) {
  if (a.beta_P_f == 0.0f)
    return quartic_root(k.alpha, rcv, k.gq, eint * rcp(rcv), 1e-7f, a.newton_max_iter, T);
  return power_root(k.alpha, 4.0f + a.beta_P_f, rcv, k.gq, eint * rcp(rcv), 1e-7f,
                    a.newton_max_iter, T);
}
// The emission term q = dt cbar rho (kP(T) B(T) + kS J~) in float.
__device__ __forceinline__ float float_q(const StepArgs<float> &a, const QuarticF &k, float T,
                                         float SI, float SG) {
  float dPT = k.dP;  // dP with kappa_P at T^{n+1}
  if (a.beta_P_f != 0.0f) dPT = k.dP * powf(T / a.T_ref_f, a.beta_P_f);
  const float B = a.a_rad_4pi_f * (T * T) * (T * T);
  const float J = fmaf(dPT * B, SG, SI) * k.rU;
  return fmaf(dPT, B, k.dS * J);
}

// q of an interior cell of a float state that the float arithmetic of
// source_q_fast could not give: power-law opacities and values out of range of
// refine_quartic take the float root refined in double by refine_root; where a
// float value is not finite or the float Newton did not converge, the double
// solve of source_q.  Returns q and the status bits.
__device__ __forceinline__ float2 source_q_double(const StepArgs<float> &a, const GasStatic &gr,
                                                  const GasDyn &gd, float SI, float SG, float S1,
                                                  float eint) {
  const QuarticF k = float_coeffs(a, gr.frkP, gr.frkJ, gr.frkS, eint, SI, SG, S1);
  float Tf;
  if (isfinite(k.alpha) && isfinite(k.gq) && !float_root(a, k, gr.frcv, eint, &Tf) &&
      isfinite(Tf)) {
    const double T = refine_root(k.alpha, a.beta_P_f, a.beta_P, gr.rcv, k.gq, Tf);
    const float q = float_q(a, k, (float)T, SI, SG);
    if (isfinite(q)) return make_float2(q, 0.0f);
  }
  unsigned bad = 0;
  const double q = source_q(a, gr, gd, (double)SI, (double)SG, (double)S1, bad);
  return make_float2((float)q, __uint_as_float(bad));
}

// The same out of line, for the kernels that refine in every lane of the cell: rare
// there, and its registers are many.  Where it is all of the float path (float_quartic
// = 1) or one lane per cell runs it (step_kernel), the call costs more than it saves:
// the registers that the ABI keeps across it spill in the loops around.  us per step
// with the call and without, 56^3 cells: 104 angles 354 and 248, 72 angles 173 and
// 154, float_quartic = 1 with 24 angles 98 and 97 (32^3 x 104: 72 and 47); quad rows
// with float_quartic = 1, 48^3 x 48: 57.4 and 55.2 (three quads a thread and more keep
// the call: 64^3 x 112 222 with it and 267 without).
static __device__ __noinline__ float2 source_q_slow(const StepArgs<float> &a, const GasStatic &gr,
                                                    const GasDyn &gd, float SI, float SG, float S1,
                                                    float eint) {
  return source_q_double(a, gr, gd, SI, SG, S1, eint);
}

// q of an interior cell in float, in every lane of the cell, from the float
// coefficients and the internal energy e - rho v^2 / 2 that the previous gas
// update left in cellv: the float root, by default refined (refine_quartic),
// with float_quartic = 1 (REFINE false) as it is.  The refined Newton stops at a
// relative change of 1e-4: it converges quadratically (e -> 1.5 e^2 at most), so
// the root is then within float rounding and the refinement squares what is
// left.  Going on to 1e-7, where source_q_slow's float Newton stops, takes at most
// two more iterations (1e8 random equations, quotients off by up to 2 ulp); so that
// newton_max_iter refuses the same cells as if it went on, the early stop counts
// only 8 iterations before the limit (StepArgs::quick_iter), and a limit below 16
// stops at 1e-7.  Returns false where source_q_slow has to take over.
template <bool REFINE>
__device__ __forceinline__ bool source_q_fast(const StepArgs<float> &a, const GasStatic &gr,
                                              float SI, float SG, float S1, float eint,
                                              float &q, unsigned &bad) {
  const QuarticF k = float_coeffs(a, gr.frkP, gr.frkJ, gr.frkS, eint, SI, SG, S1);
  if (!(k.gq >= 0.0f) || !(k.alpha >= 0.0f)) {
    bad |= ST_NONFINITE;
    return true;
  }
  float T;
  if (REFINE) {
    float Tf;
    if (a.beta_P_f != 0.0f || !isfinite(k.alpha) || !isfinite(k.gq) ||
        quartic_root(k.alpha, gr.frcv, k.gq, eint * rcp(gr.frcv), a.quick_tol, a.quick_iter, &Tf) ||
        !refine_quartic(k.alpha, gr.rcv, gr.frcv, k.gq, Tf, &T))
      return false;
    q = float_q(a, k, T, SI, SG);
    return isfinite(q);
  }
  if (!isfinite(k.alpha) || !isfinite(k.gq)) return false;
  const int nc = float_root(a, k, gr.frcv, eint, &T);
  q = float_q(a, k, T, SI, SG);
  if (!isfinite(q)) return false;
  if (nc) bad |= ST_NONCONV;
  return true;
}

// Resident threads per SM the register cap aims at: kernels with up to 5
// pairs per thread fit 1024 (64 registers), wider ones 768.
template <int PPT> constexpr int min_blocks() { return (PPT <= 5 ? 1024 : 768) / NT; }

__device__ __forceinline__ float source_q_refined(const StepArgs<float> &a, const GasStatic &gr,
                                                  const GasDyn &gd, float SI, float SG, float S1,
                                                  float eint, unsigned &bad) {
  float q = 0.0f;
  if (source_q_fast<true>(a, gr, SI, SG, S1, eint, q, bad)) return q;
  const float2 r = source_q_double(a, gr, gd, SI, SG, S1, eint);
  bad |= __float_as_uint(r.y);
  return r.x;
}

}  // namespace step
}  // namespace rt
