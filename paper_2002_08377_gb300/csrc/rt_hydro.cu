// Gas dynamics on the state's mesh, for radiation subcycled under a hydro
// step (Sec. 2: Eq. time evolution with the Euler fluxes; the Riemann-solver
// steps and the van Leer integrator of Sec. 2).
//
// The gas state is the one the radiation step exchanges energy and momentum
// with: rho (GasStatic::rho), m and the total energy density e (GasDyn).
// A hydro step
//   1. forms the primitives (rho, v, P) of every cell;
//   2. computes every face's flux once, from its first cell (left), its
//      second cell (right) and the face normal n_f (left to right): the HLLC
//      flux of Toro (Riemann Solvers and Numerical Methods for Fluid
//      Dynamics, Sec. 10.4) with Davis's wave-speed estimates, times the area
//      (hydro_flux_kernel, one thread per face);
//   3. updates every cell by the sum of its faces' fluxes in the cell's list
//      order, + for a face's first cell and - for its second
//      (hydro_update_kernel): each face's flux enters its two cells with
//      opposite signs, so mass, momentum and energy are conserved to
//      rounding, and the sum order is fixed (no atomics);
// once with the cell-centred states (order 1), or as the van Leer step
// (order 2): a half step over dt/2 with the cell-centred states, then the
// limited least-squares gradients of the half-step primitives
// (hydro_gradient_kernel: min sum A_f / |r|^2 (W_j - W_c - g . r)^2 over the
// face neighbours, r = x_j' - x_c, Barth-Jespersen limited to the range of the
// cell and its neighbours -- the reading of the gradient and limiter the
// radiation's reconstruction uses), and the full step over dt from the
// initial state with the fluxes of the primitives reconstructed at the face
// centroids.  Faces are static (the state's mesh).  Everything is double, and
// GB300's FP64 pipe (a warp's instruction takes 64 cycles of its scheduler) is
// what bounds the flux and gradient kernels: they are written for few FP64
// instructions (FMAs, reciprocals of 3 FMAs, one side's star state only,
// minima and maxima on the integer pipe).  64^3 linear-wave box, one van Leer
// step: 3.2 -> 1.43 ms.  After the update the per-cell radiation coefficients
// (rho kappa, rho c_v, 1 / rho) follow the new density (opacities per unit
// mass are kept).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "rt_internal.cuh"
#include "rt_step_common.cuh"

namespace rt {
namespace {

constexpr int kThreads = 256;

using step::key_value;
using step::order_key;
using step::quotient;
using step::rcp;

// primitive (rho, vx, vy, vz, P) of a conserved state
__device__ __forceinline__ void prim(double gamma, double rho, double mx, double my, double mz,
                                     double e, double *W) {
  const double ir = rcp(rho);
  W[0] = rho;
  W[1] = mx * ir;
  W[2] = my * ir;
  W[3] = mz * ir;
  W[4] = (gamma - 1.0) * fma(-0.5, fma(mx, W[1], fma(my, W[2], mz * W[3])), e);
}

__device__ __forceinline__ long long kmin(long long a, long long b) { return b < a ? b : a; }
__device__ __forceinline__ long long kmax(long long a, long long b) { return b > a ? b : a; }

// HLLC flux per unit area through a face with unit normal n, left state WL
// on the side n points away from; returns false for a non-positive density
// or pressure.  With q = rho (S - u), f = q / (S - S*) the star density and
// p* = P + q (S* - u) of the side K that holds the face, the flux F_K + S (U* -
// U_K) (Toro Eq. 10.39) is, by the jump conditions across S,
//   (f S*,  f S* (v + (S* - u) n) + p* n,  (E* + p*) S*),
//   E* = ((S - u) E + (S* - u) (q S* + P)) / (S - S*),
// one reciprocal instead of five divisions; a supersonic side is the same
// formula with S* = u (f = rho, p* = P, E* = E).  About 90 FP64 operations
// and two square roots (with both sides' fluxes and every quotient divided out
// it was 300).
__device__ __forceinline__ bool hllc(double gamma, const double (&WL)[5], const double (&WR)[5],
                                     const double *n, double (&F)[5]) {
  if (!(WL[0] > 0.0) || !(WL[4] > 0.0) || !(WR[0] > 0.0) || !(WR[4] > 0.0)) return false;
  const double uL = fma(WL[1], n[0], fma(WL[2], n[1], WL[3] * n[2]));
  const double uR = fma(WR[1], n[0], fma(WR[2], n[1], WR[3] * n[2]));
  const double aL = sqrt(gamma * WL[4] * rcp(WL[0])), aR = sqrt(gamma * WR[4] * rcp(WR[0]));
  // the slowest and fastest signal speeds (Davis) and the contact speed
  const double SL = fmin(uL - aL, uR - aR), SR = fmax(uL + aL, uR + aR);
  const double qL = WL[0] * (SL - uL), qR = WR[0] * (SR - uR);
  double Ss = fma(qL, uL, fma(-qR, uR, WR[4] - WL[4])) * rcp(qL - qR);
  bool left = Ss >= 0.0;  // the side of the contact that holds the face
  if (SL >= 0.0) {
    left = true;
    Ss = uL;
  } else if (SR <= 0.0) {
    left = false;
    Ss = uR;
  }
  const double S = left ? SL : SR, u = left ? uL : uR, q = left ? qL : qR;
  double w[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) w[k] = left ? WL[k] : WR[k];
  const double v2 = fma(w[1], w[1], fma(w[2], w[2], w[3] * w[3]));
  const double E = fma(0.5 * w[0], v2, w[4] * (1.0 / (gamma - 1.0)));
  const double inv = rcp(S - Ss), dS = Ss - u;
  const double G = q * inv * Ss, ps = fma(q, dS, w[4]);
  const double Es = fma(S - u, E, dS * fma(q, Ss, w[4])) * inv;
  const double gn = fma(G, dS, ps);
  F[0] = G;
#pragma unroll
  for (int d = 0; d < 3; ++d) F[1 + d] = fma(G, w[1 + d], gn * n[d]);
  F[4] = (Es + ps) * Ss;
  return true;
}

// W[c][5] from (GasStatic::rho, GasDyn) or from U[c][5] = (rho, mx, my, mz, e);
// a non-positive density or pressure is latched in status
__global__ void prim_kernel(const GasStatic *__restrict__ gs, const GasDyn *__restrict__ gd,
                            const double *__restrict__ U, int64_t n, double gamma, double *W,
                            unsigned *status, unsigned long long *bad) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n) return;
  double *w = W + 5 * c;
  if (U)
    prim(gamma, U[5 * c], U[5 * c + 1], U[5 * c + 2], U[5 * c + 3], U[5 * c + 4], w);
  else
    prim(gamma, gs[c].rho, gd[c].mx, gd[c].my, gd[c].mz, gd[c].e, w);
  if (!(w[0] > 0.0) || !(w[4] > 0.0)) {
    atomicOr(status, ST_NONFINITE);
    atomicMin(bad, (unsigned long long)c);
  }
}

// area x HLLC flux of every face, from cell-centred or reconstructed states
__global__ void __launch_bounds__(kThreads)
    flux_kernel(const HydroFace *__restrict__ faces, int64_t nf,
                            const double *__restrict__ W, const double *__restrict__ grad,
                            double gamma, double *flux, unsigned *status,
                            unsigned long long *bad) {
  const int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= nf) return;
  const HydroFace fc = faces[f];
  double WL[5], WR[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    WL[q] = W[5 * (int64_t)fc.i + q];
    WR[q] = W[5 * (int64_t)fc.j + q];
  }
  if (grad) {
    const double *gi = grad + 15 * (int64_t)fc.i, *gj = grad + 15 * (int64_t)fc.j;
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      WL[q] = fma(gi[q], fc.oi[0], fma(gi[5 + q], fc.oi[1], fma(gi[10 + q], fc.oi[2], WL[q])));
      WR[q] = fma(gj[q], fc.oj[0], fma(gj[5 + q], fc.oj[1], fma(gj[10 + q], fc.oj[2], WR[q])));
    }
  }
  double F[5];
  double *out = flux + 5 * f;
  if (!hllc(gamma, WL, WR, fc.n, F)) {
    atomicOr(status, ST_NONFINITE);
    atomicMin(bad, (unsigned long long)fc.i);
#pragma unroll
    for (int q = 0; q < 5; ++q) out[q] = 0.0;
    return;
  }
#pragma unroll
  for (int q = 0; q < 5; ++q) out[q] = fc.area * F[q];
}

// U_out = U_in - h / V sum over the cell's slots in list order of
// sign x face flux.  U_in / U_out: (rho, m, e) either as (GasStatic::rho,
// GasDyn) or as U[c][5]; rho_out may be a plain array.
//
// One thread per cell and quantity, five neighbouring threads on a cell: a face's
// five values are one run of 40 bytes to them.  (One thread per cell read each value
// at a stride: 131 us at 64^3, now 65; the additions alone take 35.)
__global__ void update_kernel(const int64_t *__restrict__ ptr, const int32_t *__restrict__ face,
                              const double *__restrict__ flux, const double *__restrict__ vol,
                              int64_t n, double h, const GasStatic *__restrict__ gs_in,
                              const GasDyn *gd_in, double *U_out, double *rho_out,
                              GasDyn *gd_out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t c = i / 5;
  const int q = (int)(i - 5 * c);
  if (c >= n) return;
  double s = 0.0;
  const int64_t k1 = ptr[c + 1];
#pragma unroll 8
  for (int64_t k = ptr[c]; k < k1; ++k) {
    const int32_t f = face[k];  // ~f: the cell is the face's second cell
    const double F = flux[5 * (int64_t)(f < 0 ? ~f : f) + q];
    // the sign as bits: a conditional negation became two additions, one of them masked
    s += __hiloint2double(__double2hiint(F) ^ (f & (int)0x80000000), __double2loint(F));
  }
  const double hv = h * rcp(vol[c]);
  // gd_out may be gd_in: a thread reads and writes its own quantity only
  const GasDyn *d = gd_in + c;
  const double u =
      *(q == 0 ? &gs_in[c].rho : q == 1 ? &d->mx : q == 2 ? &d->my : q == 3 ? &d->mz : &d->e);
  const double r = fma(-hv, s, u);
  if (U_out) {
    U_out[i] = r;
  } else {
    GasDyn *o = gd_out + c;
    *(q == 0 ? rho_out + c : q == 1 ? &o->mx : q == 2 ? &o->my : q == 3 ? &o->mz : &o->e) = r;
  }
}

// The static part of the least-squares gradients, once per state (the faces
// do not move): per slot the weight A_f / |r|^2 times r = x_f - x_c - (x_f
// - x_j'), and per cell the cofactors C and the determinant of the normal
// matrix M = sum over the slots in list order of (A_f / |r|^2) r r^T, each
// rounded as the per-step formula would round it.
__global__ void lsq_setup_kernel(const int64_t *__restrict__ ptr, HydroSlot *slot, int64_t n,
                                 double *lsq) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n) return;
  double M[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
  for (int64_t k = ptr[c]; k < ptr[c + 1]; ++k) {
    HydroSlot &sl = slot[k];
    const double r[3] = {sl.own[0] - sl.nbr[0], sl.own[1] - sl.nbr[1], sl.own[2] - sl.nbr[2]};
    const double w = sl.area / (r[0] * r[0] + r[1] * r[1] + r[2] * r[2]);
    const double wr[3] = {w * r[0], w * r[1], w * r[2]};
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      sl.wr[x] = wr[x];
#pragma unroll
      for (int y = 0; y < 3; ++y) M[x][y] += wr[x] * r[y];
    }
  }
  double *C = lsq + 10 * c;  // C[3 x + y], then the determinant
  C[0] = M[1][1] * M[2][2] - M[1][2] * M[2][1];
  C[1] = M[0][2] * M[2][1] - M[0][1] * M[2][2];
  C[2] = M[0][1] * M[1][2] - M[0][2] * M[1][1];
  C[3] = M[1][2] * M[2][0] - M[1][0] * M[2][2];
  C[4] = M[0][0] * M[2][2] - M[0][2] * M[2][0];
  C[5] = M[0][2] * M[1][0] - M[0][0] * M[1][2];
  C[6] = M[1][0] * M[2][1] - M[1][1] * M[2][0];
  C[7] = M[0][1] * M[2][0] - M[0][0] * M[2][1];
  C[8] = M[0][0] * M[1][1] - M[0][1] * M[1][0];
  C[9] = M[0][0] * C[0] + M[0][1] * C[3] + M[0][2] * C[6];
}

// Limited least-squares gradients grad[c][3][5] of the primitives W[c][5]
// (x, y, z components of the five fields): g = M^-1 b with
// b = sum A_f / |r|^2 r (W_j - W_c) over the cell's slots in list order (the
// static weights and the inverse by cofactors from lsq_setup_kernel).  Two
// passes over the cell's slots serve all five fields: the first forms the
// right-hand sides and the neighbour range, the second the extreme face
// increments g . (x_f - x_c).  The Barth-Jespersen factor min_f (hi - v) / dv
// (dv > 0) or (lo - v) / dv (dv < 0) is taken as one division by the largest
// positive and one by the most negative increment (the numerators have fixed
// signs).  The ranges are kept as order-preserving integers: a double minimum
// takes FP64 instructions.
__global__ void __launch_bounds__(kThreads, 2)
    gradient_kernel(const int64_t *__restrict__ ptr, const int32_t *__restrict__ nbr,
                    const HydroSlot *__restrict__ slot, const double *__restrict__ lsq,
                    const double *__restrict__ W, int64_t n, double *grad) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n) return;
  const int64_t k0 = ptr[c], k1 = ptr[c + 1];
  const double *Wc = W + 5 * c;
  double v[5], b[5][3];
  long long lo[5], hi[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    v[q] = Wc[q];
    lo[q] = hi[q] = order_key(v[q]);
    b[q][0] = b[q][1] = b[q][2] = 0.0;
  }
  for (int64_t k = k0; k < k1; ++k) {
    const double wr[3] = {slot[k].wr[0], slot[k].wr[1], slot[k].wr[2]};
    const double *Wj = W + 5 * (int64_t)nbr[k];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      const double vj = Wj[q], dv = vj - v[q];
#pragma unroll
      for (int x = 0; x < 3; ++x) b[q][x] = fma(wr[x], dv, b[q][x]);
      const long long kj = order_key(vj);
      lo[q] = kmin(lo[q], kj);
      hi[q] = kmax(hi[q], kj);
    }
  }
  const double *C = lsq + 10 * c;
  const double idet = rcp(C[9]);
  double g[5][3];
  long long dmax[5], dmin[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) {
#pragma unroll
    for (int x = 0; x < 3; ++x)
      g[q][x] = fma(C[3 * x], b[q][0], fma(C[3 * x + 1], b[q][1], C[3 * x + 2] * b[q][2])) * idet;
    dmax[q] = dmin[q] = 0;  // the key of 0
  }
  for (int64_t k = k0; k < k1; ++k) {
    const double o0 = slot[k].own[0], o1 = slot[k].own[1], o2 = slot[k].own[2];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      const long long kd = order_key(fma(g[q][0], o0, fma(g[q][1], o1, g[q][2] * o2)));
      dmax[q] = kmax(dmax[q], kd);
      dmin[q] = kmin(dmin[q], kd);
    }
  }
  double *out = grad + 15 * c;
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    // Barth-Jespersen: the largest factor keeping every face value in [lo, hi]
    const double up = key_value(dmax[q]), dn = key_value(dmin[q]);
    double alpha = 1.0;
    if (up > 0.0) alpha = fmin(alpha, quotient(key_value(hi[q]) - v[q], up));
    if (dn < 0.0) alpha = fmin(alpha, quotient(key_value(lo[q]) - v[q], dn));
#pragma unroll
    for (int x = 0; x < 3; ++x) out[5 * x + q] = g[q][x] * alpha;
  }
}

// The radiation's per-cell coefficients from the new density: rho kappa
// with the opacities per unit mass, rho c_v, 1 / rho and their float copies.
__global__ void refresh_kernel(const double *__restrict__ rho, const double *__restrict__ kmass,
                               int64_t n, double cv, GasStatic *gs) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n) return;
  const double r = rho[c];
  GasStatic g;
  g.rho = r;
  g.rkP = r * kmass[3 * c];
  g.rkJ = r * kmass[3 * c + 1];
  g.rkS = r * kmass[3 * c + 2];
  g.inv_rho = 1.0 / r;
  g.rcv = r * cv;
  g.frkP = (float)g.rkP;
  g.frkJ = (float)g.rkJ;
  g.frkS = (float)g.rkS;
  g.frcv = (float)g.rcv;
  gs[c] = g;
}

// cfl V^(1/3) / (|v| + sound speed), minimum over cells (positive doubles
// order as their bit patterns)
__global__ void dt_kernel(const GasStatic *__restrict__ gs, const GasDyn *__restrict__ gd,
                          const double *__restrict__ vol, int64_t n, double gamma, double cfl,
                          unsigned long long *best) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n) return;
  double W[5];
  prim(gamma, gs[c].rho, gd[c].mx, gd[c].my, gd[c].mz, gd[c].e, W);
  const double v = sqrt(W[1] * W[1] + W[2] * W[2] + W[3] * W[3]);
  const double a = sqrt(gamma * W[4] / W[0]);
  const double t = cfl * (cbrt(vol[c]) / (v + a));
  if (t > 0.0) atomicMin(best, (unsigned long long)__double_as_longlong(t));
}

unsigned grid(int64_t n) { return (unsigned)((n + kThreads - 1) / kThreads); }

}  // namespace

int hydro_setup(rt_state *s, const rt_mesh_desc *m) {
  const int64_t N = s->n_cells, Nf = m->n_faces;
  std::vector<int64_t> slot_of(N);
  for (int64_t ic = 0; ic < N; ++ic) slot_of[s->cell_of[ic]] = ic;
  // faces numbered in the order the cells (internal order) list them first, so
  // that neighbouring threads of the flux kernel gather neighbouring cells
  std::vector<int32_t> number(Nf, -1);
  {
    int32_t next = 0;
    for (int64_t ic = 0; ic < N; ++ic) {
      const int64_t c = s->cell_of[ic];
      for (int64_t k = m->cell_face_ptr[c]; k < m->cell_face_ptr[c + 1]; ++k) {
        const int32_t e = m->cell_face_idx[k];
        const int64_t f = e >= 0 ? e : -(int64_t)e - 1;
        if (number[f] < 0) number[f] = next++;
      }
    }
  }
  std::vector<HydroFace> faces(Nf);
  for (int64_t f = 0; f < Nf; ++f) {
    HydroFace &h = faces[number[f]];
    h.i = (int32_t)slot_of[m->face_cells[2 * f]];
    h.j = (int32_t)slot_of[m->face_cells[2 * f + 1]];
    h.area = m->face_area[f];
    for (int d = 0; d < 3; ++d) {
      h.n[d] = m->face_normal[3 * f + d];
      h.oi[d] = m->face_offset[6 * f + d];
      h.oj[d] = m->face_offset[6 * f + 3 + d];
    }
  }
  std::vector<HydroSlot> slots(s->nnz);
  std::vector<int32_t> ids(s->nnz);
  int64_t o = 0;
  for (int64_t ic = 0; ic < N; ++ic) {
    const int64_t c = s->cell_of[ic];
    for (int64_t k = m->cell_face_ptr[c]; k < m->cell_face_ptr[c + 1]; ++k, ++o) {
      const int32_t e = m->cell_face_idx[k];
      const int64_t f = e >= 0 ? e : -(int64_t)e - 1;
      const bool first = e >= 0;
      HydroSlot &h = slots[o];
      for (int d = 0; d < 3; ++d) {
        h.own[d] = m->face_offset[6 * f + (first ? 0 : 3) + d];
        h.nbr[d] = m->face_offset[6 * f + (first ? 3 : 0) + d];
      }
      h.area = m->face_area[f];
      ids[o] = first ? number[f] : ~number[f];
    }
  }
  cudaError_t e;
  auto up = [&](void **dst, const void *src, size_t bytes) {
    e = cudaMalloc(dst, bytes);
    if (e == cudaSuccess) e = cudaMemcpy(*dst, src, bytes, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) s->device_bytes += bytes;
    return e == cudaSuccess;
  };
  if (!up((void **)&s->d_hface, faces.data(), sizeof(HydroFace) * Nf) ||
      !up((void **)&s->d_hslot, slots.data(), sizeof(HydroSlot) * s->nnz) ||
      !up((void **)&s->d_hface_id, ids.data(), sizeof(int32_t) * s->nnz))
    return e == cudaErrorMemoryAllocation ? RT_ERR_OOM : RT_ERR_CUDA;
  e = cudaMalloc((void **)&s->d_hlsq, sizeof(double) * 10 * (size_t)N);
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? RT_ERR_OOM : RT_ERR_CUDA;
  s->device_bytes += sizeof(double) * 10 * (size_t)N;
  lsq_setup_kernel<<<grid(N), kThreads, 0, s->stream>>>(s->d_ptr, s->d_hslot, N, s->d_hlsq);
  s->launches++;
  e = cudaGetLastError();
  if (e != cudaSuccess) return RT_ERR_CUDA;
  const size_t work = sizeof(double) * ((size_t)N * (5 + 15 + 5 + 1 + 3) + (size_t)Nf * 5);
  e = cudaMalloc((void **)&s->d_hwork, work);
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? RT_ERR_OOM : RT_ERR_CUDA;
  s->device_bytes += work;
  return RT_OK;
}

// The work area: W[N][5], grad[N][15], U half step [N][5], rho [N],
// opacities per unit mass [N][3], face fluxes [Nf][5].
static double *work_W(rt_state *s) { return s->d_hwork; }
static double *work_grad(rt_state *s) { return s->d_hwork + 5 * s->n_cells; }
static double *work_U(rt_state *s) { return s->d_hwork + 20 * s->n_cells; }
static double *work_rho(rt_state *s) { return s->d_hwork + 25 * s->n_cells; }
double *hydro_kmass(rt_state *s) { return s->d_hwork + 26 * s->n_cells; }
static double *work_flux(rt_state *s) { return s->d_hwork + 29 * s->n_cells; }

cudaError_t launch_hydro_step(rt_state *s, double dt, int order) {
  const int64_t N = s->n_cells, Nf = s->n_faces;
  const double g = s->params.gamma_gas;
  double *W = work_W(s), *grad = work_grad(s), *U = work_U(s), *rho = work_rho(s);
  double *flux = work_flux(s);
  prim_kernel<<<grid(N), kThreads, 0, s->stream>>>(s->d_gs, s->d_gd, nullptr, N, g, W, s->d_status,
                                                   s->d_bad);
  flux_kernel<<<grid(Nf), kThreads, 0, s->stream>>>(s->d_hface, Nf, W, nullptr, g, flux,
                                                    s->d_status, s->d_bad);
  s->launches += 2;
  if (order == 1) {
    update_kernel<<<grid(5 * N), kThreads, 0, s->stream>>>(s->d_ptr, s->d_hface_id, flux, s->d_volume, N,
                                                       dt, s->d_gs, s->d_gd, nullptr, rho, s->d_gd);
    s->launches++;
  } else {
    // half step into U, gradients of its primitives, full step from the start
    update_kernel<<<grid(5 * N), kThreads, 0, s->stream>>>(s->d_ptr, s->d_hface_id, flux, s->d_volume, N,
                                                       0.5 * dt, s->d_gs, s->d_gd, U, nullptr,
                                                       nullptr);
    prim_kernel<<<grid(N), kThreads, 0, s->stream>>>(nullptr, nullptr, U, N, g, W, s->d_status,
                                                     s->d_bad);
    gradient_kernel<<<grid(N), kThreads, 0, s->stream>>>(s->d_ptr, s->d_nbr, s->d_hslot,
                                                         s->d_hlsq, W, N, grad);
    flux_kernel<<<grid(Nf), kThreads, 0, s->stream>>>(s->d_hface, Nf, W, grad, g, flux,
                                                      s->d_status, s->d_bad);
    update_kernel<<<grid(5 * N), kThreads, 0, s->stream>>>(s->d_ptr, s->d_hface_id, flux, s->d_volume, N,
                                                       dt, s->d_gs, s->d_gd, nullptr, rho, s->d_gd);
    s->launches += 5;
  }
  // the radiation's per-cell coefficients follow the new density, and the
  // new primitives are checked
  refresh_kernel<<<grid(N), kThreads, 0, s->stream>>>(rho, hydro_kmass(s), N,
                                                      s->params.r_gas / (g - 1.0), s->d_gs);
  prim_kernel<<<grid(N), kThreads, 0, s->stream>>>(s->d_gs, s->d_gd, nullptr, N, g, W, s->d_status,
                                                   s->d_bad);
  s->launches += 2;
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = launch_cellv(s);
  return e;
}

cudaError_t launch_hydro_dt(rt_state *s, double cfl, double *dt) {
  unsigned long long *best = reinterpret_cast<unsigned long long *>(s->d_out16);
  const unsigned long long init = 0x7ff0000000000000ull;  // +inf
  cudaError_t e = cudaMemcpyAsync(best, &init, sizeof init, cudaMemcpyHostToDevice, s->stream);
  if (e != cudaSuccess) return e;
  dt_kernel<<<grid(s->n_cells), kThreads, 0, s->stream>>>(s->d_gs, s->d_gd, s->d_volume,
                                                          s->n_cells, s->params.gamma_gas, cfl,
                                                          best);
  s->launches++;
  unsigned long long bits = 0;
  e = cudaMemcpyAsync(&bits, best, sizeof bits, cudaMemcpyDeviceToHost, s->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
  if (e == cudaSuccess) std::memcpy(dt, &bits, sizeof bits);
  return e;
}

namespace {
__global__ void density_out_kernel(const GasStatic *__restrict__ gs,
                                   const int64_t *__restrict__ cell_of, int64_t n, double *rho) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) rho[cell_of[i]] = gs[i].rho;
}
}  // namespace

cudaError_t launch_density_out(rt_state *s, double *rho) {
  density_out_kernel<<<grid(s->n_cells), kThreads, 0, s->stream>>>(s->d_gs, s->d_cell_of,
                                                                   s->n_cells, rho);
  s->launches++;
  return cudaGetLastError();
}

}  // namespace rt
