// The fused radiation step of double states: upwind transport (Sec. 2.2) and
// the implicit comoving source update with gas exchange (Sec. 2.3), boundary
// (Sec. 2.4) and emitter cells (Sec. 2.5), one kernel per step.
//
// Blocks of 32 cells x 8 threads over the pair layout (thread `sub` owns the
// pairs sub + 8 j), the phases of the float kernel (rt_step.cu).  GB300 issues
// a warp's FP64 instruction over 64 cycles of its scheduler, so the kernel is
// bound by the number of FP64 instructions and everything else hides behind
// them.  Where they go, per pair, on a static mesh:
//   1 per face (face_sum_static64), 4 for I*, 35 for phase A, 16 for phase C:
//   phase A keeps z = Gamma^3 I*, r = 1 / (Gamma^3 (1 + x Gamma)) and x Gamma
//   in registers, so phase C forms no direction cosines and no reciprocal;
//   a reciprocal is 3 operations (rcp);
//   the four sums of a cell reduce over its 8 threads by 4 adds (cell_reduce4);
//   the lane-per-cell phases B and D run on a warp that rotates with the
//   block, so that they load the SM's four schedulers evenly.
// One step of the 64^3 shadows box with 80 angles: 1.65 ms (2.38 ms with two
// FMAs per face and pair and 86 operations per pair in the source).
#include <cuda_runtime.h>

#include "rt_internal.cuh"
#include "rt_step_args.cuh"

namespace rt {
namespace {
using namespace step;

struct Shared64 {
  double sum[4][CPB];  // phase A: S_I, S_G, S_1; phase C: sum w dI, sum w n dI
  double q[CPB];       // dt cbar rho (kP B + kS J) per interior cell
  unsigned bad[CPB];
};

// The sums of v0..v3 over a cell's 8 threads: thread `sub` returns that of
// v[sub / 2] (the same tree as four butterflies over lanes 4, 2, 1).
__device__ __forceinline__ double cell_reduce4(double v0, double v1, double v2, double v3,
                                               int sub) {
  const bool hi = sub & 4, odd = sub & 2;
  double a = hi ? v2 : v0, b = hi ? v3 : v1;
  a += __shfl_xor_sync(0xffffffffu, hi ? v0 : v2, 4);
  b += __shfl_xor_sync(0xffffffffu, hi ? v1 : v3, 4);
  double c = odd ? b : a;
  c += __shfl_xor_sync(0xffffffffu, odd ? a : b, 2);
  c += __shfl_xor_sync(0xffffffffu, c, 1);
  return c;
}

template <typename M, bool MOVING>
__global__ void __launch_bounds__(NT, 2) step64_kernel(const StepArgs<double> a) {
  using V = double2;
  constexpr int PPT = M::PPT;
  __shared__ Shared64 sh;
  __shared__ SharedGas gas;
  const int64_t tile = blockIdx.x;
  const int lc = threadIdx.x / KT;
  const int sub = threadIdx.x % KT;
  const int64_t cell = tile * CPB + lc;
  const bool live = cell < a.n_cells;
  const int64_t c = live ? cell : a.n_cells - 1;  // dead lanes shadow the last cell
  const int RS = a.row;
  const int np = M::count(a.half, sub);

  // lane-per-cell phases: lanes of warp wb (phase B) and wd (phase D), one cell each
  const int warp = threadIdx.x / 32, lp = threadIdx.x % 32;
  const int wb = (int)(tile % (NT / 32)), wd = (wb + 2) % (NT / 32);
  const int64_t cl = tile * CPB + lp;
  if (warp == wb && cl < a.n_cells) {
    // prefetch of the cells' gas state for phases B and D
    const char *g = reinterpret_cast<const char *>(a.gs + cl);
    const char *d = reinterpret_cast<const char *>(a.gd + cl);
#pragma unroll
    for (int k = 0; k < 4; ++k)
      cp_async16(reinterpret_cast<char *>(&gas.gs[lp]) + 16 * k, g + 16 * k);
#pragma unroll
    for (int k = 0; k < 2; ++k)
      cp_async16(reinterpret_cast<char *>(&gas.gd[lp]) + 16 * k, d + 16 * k);
  }

  // ---------------- transport, I* = I - dt/V sum_f u I_up
  double Ia[PPT], Ib[PPT];
  M::load(a.I_in + (size_t)c * RS, sub, Ia, Ib, np);
  if (!a.src_only) {
    double acca[PPT], accb[PPT];
#pragma unroll
    for (int j = 0; j < PPT; ++j) acca[j] = accb[j] = 0.0;
    const double none[PPT] = {};  // double faces read tabulated coefficients, no directions
    face_sum<double, M, MOVING, false, TRANSPORT_FORWARD>(
        a.slot, a.nbr, a.wface, a.uface, a.half, a.ptr[c], a.ptr[c + 1], a.I_in, RS, sub, none,
        none, none, Ia, Ib, acca, accb, np, a.kout ? a.kout + (size_t)c * RS : nullptr);
    const double dtv = a.dt * a.inv_vol[c];
#pragma unroll
    for (int j = 0; j < PPT; ++j) {
      Ia[j] = fma(-dtv, acca[j], Ia[j]);  // I*
      Ib[j] = fma(-dtv, accb[j], Ib[j]);
    }
    if constexpr (MOVING) {
      // geometric conservation law: V^{n+1} I* = V^n I - dt sum_f u I_up, i.e.
      // the fixed-volume I* times V^n / V^{n+1} = 1 / (1 + dt rate / V^n)
      if (a.gcl_rate) {
        const double ratio = rcp(fma(dtv, a.gcl_rate[c], 1.0));
#pragma unroll
        for (int j = 0; j < PPT; ++j) {
          Ia[j] *= ratio;
          Ib[j] *= ratio;
        }
      }
    }
  }

  // ---------------- phase A: the comoving frame (see the float kernel): per
  // angle Gamma = 1 -+ v.n / c, and with r = 1 / (Gamma^3 (1 + x Gamma)),
  // z = Gamma^3 I*, t = w Gamma r the sums S_1 = sum t, S_G = sum t Gamma,
  // S_I = sum t Gamma z.  Emitter cells take their own rate in x (their sums
  // are unused).
  const int kind = a.kind[c];
  const double icr = a.inv_c_r;
  const double vx = a.cellv[4 * c] * icr, vy = a.cellv[4 * c + 1] * icr,
               vz = a.cellv[4 * c + 2] * icr;
  double xs, q = 0.0;  // x / Gamma; q: the emission term of phase C
  double2 ax = make_double2(0.0, 0.0);
  if (kind != RT_CELL_INTERIOR) ax = a.aux[c];
  if (kind == RT_CELL_EMITTER)
    xs = a.dt * a.cbar * ax.x;
  else
    xs = a.dt_cbar_r * (a.gs[c].rkJ + a.gs[c].rkS);
  const double gam = frame_gamma(a.boost, vx, vy, vz);
  if (a.boost) xs *= gam;
  const V *W2 = reinterpret_cast<const V *>(a.wt2);
  double ra[PPT], rb[PPT], xga[PPT], xgb[PPT];
  double sI = 0.0, sG = 0.0, s1 = 0.0;
  if (kind != RT_CELL_BOUNDARY) {
    const V XS = mk(xs, xs), one = mk(1.0, 1.0);
    V sIv = mk(0.0, 0.0), sGv = sIv, s1v = sIv;  // unnormalised: cancels in phase B
#pragma unroll
    for (int j = 0; j < PPT; ++j) {
      const int p = (M::FULL || j < np) ? M::pair(j, sub) : 0;
      double nx, ny, nz;
      load_dir(a.dir, p, nx, ny, nz);
      const double bn = fma(vx, nx, fma(vy, ny, vz * nz));
      const V G = mk(1.0 - bn, 1.0 + bn);
      const V G3 = pmul(pmul(G, G), G), XG = pmul(XS, G);
      const V r = prcp<double>(pmul(G3, padd(XG, one)));
      const V z = pmul(mk(Ia[j], Ib[j]), G3);
      if (M::FULL || j < np) {
        const V t = pmul(pmul(W2[p], r), G), tG = pmul(t, G);
        s1v = padd(s1v, t);
        sGv = padd(sGv, tG);
        sIv = pfma(tG, z, sIv);
      }
      Ia[j] = z.x;
      Ib[j] = z.y;
      ra[j] = r.x;
      rb[j] = r.y;
      xga[j] = XG.x;
      xgb[j] = XG.y;
    }
    sI = sIv.x + sIv.y;
    sG = sGv.x + sGv.y;
    s1 = s1v.x + s1v.y;
  }
  {
    const double v = cell_reduce4(sI, sG, s1, 0.0, sub);
    if (!(sub & 1)) sh.sum[sub / 2][lc] = v;
  }
  if (warp == wb) cp_async_wait_all();
  __syncthreads();

  // ---------------- phase B: the temperature quartic, one lane per cell.  To
  // all orders Gamma = gamma G: S_I -> gamma^4 S_I, S_G -> gamma S_G here and
  // q -> q / gamma^3 in phase C (gamma = 1: exact).
  if (warp == wb) {
    double ql = 0.0;
    unsigned bl = 0;
    if (cl < a.n_cells && a.kind[cl] == RT_CELL_INTERIOR) {
      double SI = sh.sum[0][lp], SG = sh.sum[1][lp];
      if (a.boost) {
        const double g = frame_gamma(a.boost, a.cellv[4 * cl] * icr, a.cellv[4 * cl + 1] * icr,
                                     a.cellv[4 * cl + 2] * icr);
        SI *= (g * g) * (g * g);
        SG *= g;
      }
      ql = source_q(a, gas.gs[lp], gas.gd[lp], SI, SG, sh.sum[2][lp], bl);
    }
    sh.q[lp] = ql;
    sh.bad[lp] = bl;
  }
  __syncthreads();

  // ---------------- phase C: new intensities and the radiation change.
  // Interior: I' = (z + q) r, and the change I* - I' as the source term itself,
  // (z x Gamma - q) r, whose rounding is relative to the change, not to I*;
  // emitters the same with their rate in x and q = rate I_src; boundary:
  // I' = I* - f (I* - I0), the change f (I* - I0).
  double de = 0.0, dfx = 0.0, dfy = 0.0, dfz = 0.0;
  {
    if (kind == RT_CELL_BOUNDARY) {
      const double f = (ax.x <= a.dt) ? 1.0 : a.dt / ax.x;
      double tx[PPT], ty[PPT];
      M::load(a.I0 + (size_t)a.bc_row[c] * RS, sub, tx, ty, np);
#pragma unroll
      for (int j = 0; j < PPT; ++j) {
        const double da = Ia[j] - tx[j], db = Ib[j] - ty[j];
        Ia[j] = fma(-f, da, Ia[j]);
        Ib[j] = fma(-f, db, Ib[j]);
        ra[j] = f * da;
        rb[j] = f * db;
      }
    } else {
      q = kind == RT_CELL_EMITTER ? xs * ax.y : sh.q[lc];
      if (a.boost) q /= kind == RT_CELL_EMITTER ? (gam * gam) * (gam * gam) : gam * gam * gam;
#pragma unroll
      for (int j = 0; j < PPT; ++j) {
        const double da = fma(Ia[j], xga[j], -q) * ra[j], db = fma(Ib[j], xgb[j], -q) * rb[j];
        Ia[j] = (Ia[j] + q) * ra[j];
        Ib[j] = (Ib[j] + q) * rb[j];
        ra[j] = da;
        rb[j] = db;
      }
    }
    if (live) M::store(a.I_out + (size_t)c * RS, sub, Ia, Ib, np);
    V dev = mk(0.0, 0.0);
#pragma unroll
    for (int j = 0; j < PPT; ++j) {
      if (M::FULL || j < np) {
        const int p = M::pair(j, sub);
        const V d = pmul(W2[p], mk(ra[j], rb[j]));
        dev = padd(dev, d);
        const double df = d.x - d.y;  // the antipode has direction -n
        double ux, uy, uz;
        load_dir(a.dir, p, ux, uy, uz);
        dfx = fma(ux, df, dfx);
        dfy = fma(uy, df, dfy);
        dfz = fma(uz, df, dfz);
      }
    }
    de = dev.x + dev.y;
  }
  {
    const double v = cell_reduce4(de, dfx, dfy, dfz, sub);
    if (!(sub & 1)) sh.sum[sub / 2][lc] = v;
  }
  __syncthreads();

  // ---------------- phase D: gas exchange (Eqs. gas1, gas2), one lane per cell
  if (warp == wd && cl < a.n_cells) {
    // a non-finite new intensity makes its weighted change, and so the
    // cell's sum, non-finite (the weights are positive)
    unsigned bad = sh.bad[lp];
    if (!isfinite(sh.sum[0][lp])) bad |= ST_NONFINITE;
    gas_exchange<double, MOVING>(a, cl, gas.gs[lp], gas.gd[lp], sh.sum[0][lp], sh.sum[1][lp],
                                 sh.sum[2][lp], sh.sum[3][lp], bad);
  }
}

template <typename M, bool MOVING>
cudaError_t launch64(rt_state *s, double dt, const StepIO &io) {
  const StepArgs<double> a = step_args<double>(s, dt, io);
  const unsigned blocks = (unsigned)((s->n_cells + CPB - 1) / CPB);
  step64_kernel<M, MOVING><<<blocks, NT, 0, s->stream>>>(a);
  s->launches++;
  return cudaGetLastError();
}

template <bool MOVING, bool FULL>
cudaError_t dispatch64(rt_state *s, double dt, const StepIO &io) {
  switch ((s->n_angles / 2 + KT - 1) / KT) {
    case 1: return launch64<PairMap<double, 1, FULL>, MOVING>(s, dt, io);
    case 2: return launch64<PairMap<double, 2, FULL>, MOVING>(s, dt, io);
    case 3: return launch64<PairMap<double, 3, FULL>, MOVING>(s, dt, io);
    case 4: return launch64<PairMap<double, 4, FULL>, MOVING>(s, dt, io);
    case 5: return launch64<PairMap<double, 5, FULL>, MOVING>(s, dt, io);
    case 6: return launch64<PairMap<double, 6, FULL>, MOVING>(s, dt, io);
    case 7: return launch64<PairMap<double, 7, FULL>, MOVING>(s, dt, io);
    case 8: return launch64<PairMap<double, 8, FULL>, MOVING>(s, dt, io);
    default: return cudaErrorInvalidValue;
  }
}

// U[k][p] = the double flux coefficient of pair p through directed face k,
// exactly the expression slot_dot evaluates (cbar A ((n_x n_fx + n_y n_fy) +
// n_z n_fz), rounded in that order): the mesh is fixed for a state's
// lifetime, so the FP64 face loop reads it instead of recomputing it.
__global__ void uface_kernel(const SlotD *__restrict__ slot, const double *__restrict__ dir,
                             int64_t nnz, int H, double *__restrict__ U) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nnz * H) return;
  const int64_t k = i / H;
  const int p = (int)(i % H);
  U[i] = slot_dot(dir[4 * p], dir[4 * p + 1], dir[4 * p + 2], load_slot<double>(slot + k));
}

// K[c][2 p + s] = sum over the cell's faces, in slot order, of max(u, 0) of
// angle p (s = 0) and of its antipode (s = 1).
__global__ void kout_kernel(const int64_t *__restrict__ ptr, const double *__restrict__ U,
                            int64_t n, int H, double2 *__restrict__ K) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n * H) return;
  const int64_t c = i / H;
  const int p = (int)(i % H);
  double ka = 0.0, kb = 0.0;
  for (int64_t k = ptr[c]; k < ptr[c + 1]; ++k) {
    const double d = U[(size_t)k * H + p];
    if (d > 0.0)
      ka += d;
    else
      kb -= d;
  }
  K[i] = make_double2(ka, kb);
}

}  // namespace

cudaError_t build_uface(rt_state *s) {
  const int H = s->n_angles / 2;
  const size_t n = (size_t)s->nnz * H;
  if (!s->d_uface) {
    cudaError_t e = cudaMalloc(&s->d_uface, n * sizeof(double));
    if (e != cudaSuccess) return e;
    s->device_bytes += n * sizeof(double);
  }
  const unsigned blocks = (unsigned)((n + 255) / 256);
  uface_kernel<<<blocks, 256, 0, s->stream>>>(reinterpret_cast<const SlotD *>(s->d_slot),
                                              reinterpret_cast<const double *>(s->d_dir), s->nnz, H,
                                              s->d_uface);
  s->launches++;
  return cudaGetLastError();
}

cudaError_t build_kout(rt_state *s) {
  const int H = s->n_angles / 2;
  const size_t n = (size_t)s->n_cells * H;
  // only where the state's later allocations (the adjoint's ten intensity
  // arrays, host-I/O staging) fit beside it
  size_t free_bytes = 0, total = 0;
  cudaError_t e = cudaMemGetInfo(&free_bytes, &total);
  if (e != cudaSuccess) return e;
  if (free_bytes / 16 < n * sizeof(double2)) return cudaSuccess;
  e = cudaMalloc(&s->d_kout, n * sizeof(double2));
  if (e != cudaSuccess) {
    s->d_kout = nullptr;
    if (e != cudaErrorMemoryAllocation) return e;
    (void)cudaGetLastError();
    return cudaSuccess;
  }
  s->device_bytes += n * sizeof(double2);
  kout_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s->stream>>>(
      s->d_ptr, s->d_uface, s->n_cells, H, reinterpret_cast<double2 *>(s->d_kout));
  s->launches++;
  return cudaGetLastError();
}

cudaError_t launch_step_io64(rt_state *s, double dt, const StepIO &io) {
  const bool full = (s->n_angles / 2) % KT == 0;
  if (s->moving)
    return full ? dispatch64<true, true>(s, dt, io) : dispatch64<true, false>(s, dt, io);
  return full ? dispatch64<false, true>(s, dt, io) : dispatch64<false, false>(s, dt, io);
}

}  // namespace rt
