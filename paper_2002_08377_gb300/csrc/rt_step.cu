// Fused radiation step of float states: upwind transport (Sec. 2.2) + implicit comoving
// source update with gas exchange (Sec. 2.3), boundary cells (Sec. 2.4) and
// emitter cells (Sec. 2.5), one kernel per step.
//
// Layout: the intensity row of a cell stores the A/2 antipodal pairs
// (angle p, angle p + A/2) together.  The flux coefficient of the antipode
// through a face is u(p + A/2) = -(n_p . s) - w, so one dot product serves both
// angles; on a static mesh exactly one of the two is inflow.
//
// quad_step_kernel (rows in the quad layout: A a multiple of 16, A >= 32) is the
// production kernel; step_kernel (rt_step_tile.cuh's PairMap) takes every other
// row.  Block = 32 cells x 8 threads.  Phases:
//   transport  all threads: the cell's faces in slot order (no atomics,
//      deterministic);
//   A  comoving weights and the angular sums of Eq. (Jcom), reduced over the
//      cell's 8 threads with shuffles;
//   B  the gas temperature quartic (source_q_fast), in every lane of the cell;
//   C  new intensities, store, radiation change per cell;
//   D  after the block's one barrier, one lane per cell: gas energy / momentum
//      (or tally) update in double (Eqs. gas1, gas2), on a warp that rotates
//      with the block.
// What bounds it: latency.  A block's time is the sum of its phases' waits (its
// stage, the gathers of the neighbour rows from L1 / L2, the double gas update),
// which four resident blocks overlap only in part: no unit is saturated (96^3 x
// 80: issue 59 %, L1 data pipe 62 %, DRAM 24 %, FP64 10 %; of the 12 cycles between a
// warp's instructions 4.5 wait for loads, 1.9 for results, 1.5 at the barrier).  Hence
// the L2 prefetch one wave ahead (11 %), one block barrier only, packed FP32 on (p, p+1)
// throughout, registers capped at 64 so that four blocks fit, and L1 given what shared
// memory leaves.  Per step, before (double refinement between two barriers, no
// prefetch) and now, rows bit for bit the same: 96^3 x 80 static 558 -> 493 us,
// 128^3 x 80 1290 -> 1131, 64^3 x 96 211 -> 168, 100^3 x 48 moving 511 -> 484.
// Staging every row a tile reads in shared memory by bulk copies (128^3 x 64:
// 1.18 against 0.93 ms) and 4 threads a cell (the same time) did not pay.
#include <cuda_runtime.h>

#include "rt_internal.cuh"
#include "rt_step_args.cuh"
#include "rt_step_quad.cuh"
#include "rt_step_source.cuh"

namespace rt {
namespace {
using namespace step;

// Per-block sums exchanged between the phases.
struct Shared {
  float sI[CPB], sG[CPB], s1[CPB];  // the sums of Eq. (Jcom) and sum w~/(1+x), unnormalised
  float q[CPB];                     // dt cbar rho (kP B + kS J) per interior cell
  float dE[CPB], dF[3][CPB];        // sum w (I* - I') and sum w n (I* - I')
  unsigned bad[CPB];
};

// One block of CPB cells of a state whose rows are in the pair layout: the
// phases of the quad kernel, slots read from global memory, the temperature refined by
// one lane per cell between two block barriers (source_q_refined; float_quartic = 1: the
// float root in every lane, no barrier).
template <typename M, bool MOVING>
__global__ void __launch_bounds__(NT, min_blocks<M::PPT>()) step_kernel(const StepArgs<float> a) {
  __shared__ Shared sh;
  __shared__ SharedGas gas;
  const int64_t tile = blockIdx.x;
  using R = float;
  using V = float2;
  constexpr int PPT = M::PPT;
  const int lc = threadIdx.x / KT;
  const int sub = threadIdx.x % KT;
  const int64_t cell = tile * CPB + lc;
  const bool live = cell < a.n_cells;
  const int64_t c = live ? cell : a.n_cells - 1;  // dead lanes shadow the last cell
  const int RS = a.row;  // reals between intensity rows
  const int np = M::count(a.half, sub);

  // lane-per-cell phases: thread t < CPB (the first CPB / 32 warps) takes cell t
  const int lp = threadIdx.x;
  const bool lpc = lp < CPB;
  const int64_t cl = tile * CPB + lp;
  if (lpc && cl < a.n_cells) {
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

  // ---------------- phase A: transport, I* = I - dt/V sum_f u I_up
  R nx[PPT], ny[PPT], nz[PPT], Ia[PPT], Ib[PPT], acca[PPT], accb[PPT];
  M::load(a.I_in + (size_t)c * RS, sub, Ia, Ib, np);
#pragma unroll
  for (int j = 0; j < PPT; ++j) {
    load_dir(a.dir, (M::FULL || j < np) ? M::pair(j, sub) : 0, nx[j], ny[j], nz[j]);
    acca[j] = R(0);
    accb[j] = R(0);
  }
  if (!a.src_only)
    face_sum<R, M, MOVING, false, TRANSPORT_FORWARD>(
        reinterpret_cast<const SlotF *>(a.slot), a.nbr, a.wface, a.uface, a.half, a.ptr[c],
        a.ptr[c + 1], a.I_in, RS, sub, nx, ny, nz, Ia, Ib, acca, accb, np, nullptr);
  {
    const R dtv = a.dt_r * a.inv_vol[c];
#pragma unroll
    for (int j = 0; j < PPT; ++j) {
      Ia[j] = fma(-dtv, acca[j], Ia[j]);  // I*
      Ib[j] = fma(-dtv, accb[j], Ib[j]);
    }
    if constexpr (MOVING) {
      // geometric conservation law (volumes change only on a moving mesh):
      // V^{n+1} I* = V^n I - dt sum_f u I_up, i.e. the fixed-volume I* times
      // V^n / V^{n+1} = 1 / (1 + dt rate / V^n)
      if (a.gcl_rate && !a.src_only) {
        const R ratio = rcp(fma(dtv, R(a.gcl_rate[c]), R(1)));
#pragma unroll
        for (int j = 0; j < PPT; ++j) {
          Ia[j] *= ratio;
          Ib[j] *= ratio;
        }
      }
    }
  }

  // comoving frame (first order in v/c): Gamma = 1 -+ v.n / c, and the
  // angular sums of Eq. (Jcom): w~ = w / Gamma^2 (normalised by their sum),
  // S_I = sum w~ Gamma^4 I* / (1 + x Gamma), S_G = sum w~ Gamma / (1 + x Gamma).
  // To all orders Gamma = gamma G with G = 1 -+ v.n / c: the weights'
  // normalisation cancels gamma^2, so gamma enters only per cell -- x = (xs
  // gamma) G, S_I -> gamma^4 S_I, S_G -> gamma S_G (S_1 unchanged) and, in
  // phase C, q -> q / gamma^3 (emitters: rate gamma, source / gamma^4).
  // With gamma = 1 these scalings are exact.
  const int kind = a.kind[c];
  const R icr = a.inv_c_r;
  const R vxc = a.cellv[4 * c] * icr, vyc = a.cellv[4 * c + 1] * icr,
          vzc = a.cellv[4 * c + 2] * icr;
  R xs, eint = a.cellv[4 * c + 3];  // dt cbar rho (kJ + kS), internal energy
  const float4 gf = __ldg(reinterpret_cast<const float4 *>(&a.gs[c].frkP));
  const R fkP = gf.x, fkJ = gf.y, fkS = gf.z, fcv = gf.w;
  xs = a.dt_cbar_r * (fkJ + fkS);
  if (a.boost) xs *= frame_gamma(a.boost, vxc, vyc, vzc);
  const V *W2 = reinterpret_cast<const V *>(a.wt2);  // (w_p, w_{p+H})
  const V one = mk(R(1), R(1)), XS = mk(xs, xs);
  // Gamma = (1 - bn, 1 + bn) for the pair, bn = v . n_p / c; the directions
  // are read again in phase C rather than held across phase B
  V sIv = mk(R(0), R(0)), sGv = sIv, s1v = sIv;  // unnormalised: cancels in phase B
#pragma unroll
  for (int j = 0; j < PPT; ++j) {
    if (M::FULL || j < np) {
      // t = w / (Gamma^2 (1 + x Gamma)): one reciprocal per angle
      const R bn = fma(vxc, nx[j], fma(vyc, ny[j], vzc * nz[j]));
      const V G = mk(R(1) - bn, R(1) + bn);
      const V G2 = pmul(G, G);
      const V t = pmul(W2[M::pair(j, sub)], prcp<R>(pmul(G2, pfma(XS, G, one))));
      s1v = padd(s1v, t);
      sIv = pfma(pmul(t, pmul(G2, G2)), mk(Ia[j], Ib[j]), sIv);
      sGv = pfma(t, G, sGv);
    }
  }
  R sI = sIv.x + sIv.y, sG = sGv.x + sGv.y, s1 = s1v.x + s1v.y;
  sI = cell_sum(sI);
  sG = cell_sum(sG);
  s1 = cell_sum(s1);
  if (a.boost) {
    const R g = frame_gamma(a.boost, vxc, vyc, vzc), g2 = g * g;
    sI *= g2 * g2;
    sG *= g;
  }

  // ---------------- phase B: temperature quartic
  R q = 0;           // dt cbar rho (kP B + kS J~) of an interior cell
  unsigned bad = 0;  // status bits of the cell
  // float_quartic: in float, in every lane
  if (a.float_quartic) {
    // every lane of the cell solves the cell's quartic in float (the sums
    // are already in all 8 lanes), no block barrier
    if (kind == RT_CELL_INTERIOR)
      if (!source_q_fast<false>(a, a.gs[c], sI, sG, s1, eint, q, bad)) {
        const float2 r = source_q_double(a, a.gs[c], a.gd[c], sI, sG, s1, eint);
        q = r.x;
        bad |= __float_as_uint(r.y);
      }
  } else {
    // one lane per cell, between two block barriers
    if (sub == 0) {
      sh.sI[lc] = sI;
      sh.sG[lc] = sG;
      sh.s1[lc] = s1;
    }
    if (lpc) cp_async_wait_all();
    __syncthreads();
    if (lpc) {
      float ql = 0.0f;
      unsigned bl = 0;
      if (cl < a.n_cells && a.kind[cl] == RT_CELL_INTERIOR)
        ql = source_q_refined(a, gas.gs[lp], gas.gd[lp], sh.sI[lp], sh.sG[lp], sh.s1[lp],
                              a.cellv[4 * cl + 3], bl);
      sh.q[lp] = ql;
      sh.bad[lp] = bl;
    }
    __syncthreads();
    q = sh.q[lc];
    bad = sh.bad[lc];
  }

  // ---------------- phase C: new intensities and the radiation change
  R de = 0, dfx = 0, dfy = 0, dfz = 0;
  unsigned nonfinite = 0;
  {
    // boundary: I' = I* - (I* - I0) f; interior: I~' = (I~ + q Gamma) / (1 + x Gamma),
    // i.e. I' = (I* + q / Gamma^3) / (1 + x Gamma); emitter: the same with
    // x -> dt cbar (rho kappa)_src and q -> that rate times I_src (Sec. 2.5).
    // The radiation change I* - I' that the gas receives is the difference
    // of the stored intensities: the energy bookkeeping is then exact in
    // float (double states take the source term itself).
    R na[PPT], nb[PPT];
    if (kind == RT_CELL_BOUNDARY) {
      const double2 ax = a.aux[c];
      const R f = R((ax.x <= a.dt) ? 1.0 : a.dt / ax.x);
      R tx[PPT], ty[PPT];
      M::load(a.I0 + (size_t)a.bc_row[c] * RS, sub, tx, ty, np);
#pragma unroll
      for (int j = 0; j < PPT; ++j) {
        na[j] = fma(-f, Ia[j] - tx[j], Ia[j]);
        nb[j] = fma(-f, Ib[j] - ty[j], Ib[j]);
      }
    } else {
      R qq, xx = xs;
      if (kind == RT_CELL_EMITTER) {
        const double2 ax = a.aux[c];
        xx = R(a.dt * a.cbar * ax.x);
        qq = xx * R(ax.y);
        if (a.boost) {
          const R g = frame_gamma(a.boost, vxc, vyc, vzc), g2 = g * g;
          xx *= g;
          qq = xx * R(ax.y) / (g2 * g2);
        }
      } else {
        qq = q;
        if (a.boost) {
          const R g = frame_gamma(a.boost, vxc, vyc, vzc);
          qq = q / (g * g * g);
        }
      }
      const V XX = mk(xx, xx), QQ = mk(qq, qq);
#pragma unroll
      for (int j = 0; j < PPT; ++j) {
        // I' = (I* Gamma^3 + q) / (Gamma^3 (1 + x Gamma))
        R ux, uy, uz;
        load_dir(a.dir, (M::FULL || j < np) ? M::pair(j, sub) : 0, ux, uy, uz);
        const R bn = fma(vxc, ux, fma(vyc, uy, vzc * uz));
        const V G = mk(R(1) - bn, R(1) + bn);
        const V G3 = pmul(pmul(G, G), G);
        const V n = pmul(pfma(mk(Ia[j], Ib[j]), G3, QQ), prcp<R>(pmul(G3, pfma(XX, G, one))));
        na[j] = n.x;
        nb[j] = n.y;
      }
    }
    if (live) M::store(a.I_out + (size_t)c * RS, sub, na, nb, np);
    V dev = mk(R(0), R(0));
#pragma unroll
    for (int j = 0; j < PPT; ++j) {
      if (M::FULL || j < np) {
        const int p = M::pair(j, sub);
        const V d = pmul(W2[p], psub(mk(Ia[j], Ib[j]), mk(na[j], nb[j])));
        dev = padd(dev, d);
        const R df = d.x - d.y;  // the antipode has direction -n
        R ux, uy, uz;
        load_dir(a.dir, p, ux, uy, uz);
        dfx = fma(ux, df, dfx);
        dfy = fma(uy, df, dfy);
        dfz = fma(uz, df, dfz);
      }
    }
    de = dev.x + dev.y;
    // a non-finite new intensity makes its weighted change, and so de,
    // non-finite (the weights are positive)
    if (!isfinite(de)) nonfinite = ST_NONFINITE;
  }
  de = cell_sum(de);
  dfx = cell_sum(dfx);
  dfy = cell_sum(dfy);
  dfz = cell_sum(dfz);
  nonfinite = cell_or(nonfinite);
  if (sub == 0) {
    sh.dE[lc] = de;
    sh.dF[0][lc] = dfx;
    sh.dF[1][lc] = dfy;
    sh.dF[2][lc] = dfz;
    sh.bad[lc] = bad | nonfinite;
  }
  if (lpc) cp_async_wait_all();
  __syncthreads();

  // ---------------- phase D: gas exchange (Eqs. gas1, gas2), one lane per cell
  if (lpc && cl < a.n_cells)
    gas_exchange<float, MOVING>(a, cl, gas.gs[lp], gas.gd[lp], sh.dE[lp], sh.dF[0][lp], sh.dF[1][lp],
                                sh.dF[2][lp], sh.bad[lp]);
}


struct QuadShared {
  float sum[4][CPB];  // phase C: sum w dI, sum w n dI
  float q[CPB];       // power-law opacities: the emission term
  unsigned bad[CPB];
};

// Resident threads per SM the register cap aims at; SMALL: meshes of at most two
// blocks per SM (one wave at 128 registers), where the registers go into more loads
// in flight.  Such a step is a chain of load latencies: us per step without / with
// it 7.4 / 5.8 (16^3 cells x 48 angles), 9.0 / 6.8 (12^3 x 80), 18.8 / 11.1 (20^3 x
// 128), 10.7 / 9.3 (16^3 x 96, moving); beyond one wave the halved residency costs
// more than it gives.
template <int NQ, bool TAIL, bool SMALL> constexpr int quad_blocks() {
  return (SMALL ? 512 : 2 * NQ + (TAIL ? 1 : 0) <= 5 ? 1024 : 768) / NT;
}
// Faces in flight per thread of a SMALL launch (what 128 registers hold).
template <int NQ> constexpr int quad_chunk() { return NQ == 1 ? 8 : NQ == 2 ? 5 : 3; }

// The warp that does a block's lane-per-cell double work. It rotates with the block, so
// that the SM's four schedulers share that work; in a ragged last block it is one that
// has cells.
__device__ __forceinline__ int cell_warp(int64_t tile, int64_t n_cells) {
  const int w = (int)(tile % KT);
  return tile * CPB + w * (32 / KT) < n_cells ? w : 0;
}

// NQ quads and, with TAIL, one pair per thread; KT threads per cell.  REFINE: the
// float temperature root is refined (float_quartic = 0).
template <int NQ, bool TAIL, bool MOVING, bool REFINE, bool SMALL>
__global__ void __launch_bounds__(NT, quad_blocks<NQ, TAIL, SMALL>())
    quad_step_kernel(const __grid_constant__ StepArgs<float> a, const QuadDir qd, int cap) {
  constexpr int CW = 32 / KT;  // cells per warp
  __shared__ QuadShared sh;
  extern __shared__ __align__(128) unsigned char dyn[];
  const int64_t tile = blockIdx.x;
  const StageView stage = stage_at(dyn, cap, MOVING);
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
  const int lc = threadIdx.x / KT, sub = threadIdx.x % KT;
  const int64_t cell = tile * CPB + lc;
  const bool live = cell < a.n_cells;
  const int64_t c = live ? cell : a.n_cells - 1;  // dead lanes shadow the last cell
  const int RS = a.row;

  // A SMALL kernel may start while the one before it in the stream runs its last
  // phase (programmatic dependent launch): what no kernel writes (slots, the
  // connectivity, kinds, directions) is loaded first, the wait comes before
  // anything a kernel writes.  Blocks let the next kernel start once their rows are
  // stored: at their start instead, the next kernel's blocks took slots and issue
  // from this one's (16^3 cells x 48 angles 6.8 us per step, so 5.8, without 6.2).
  // On larger meshes the same displacement costs more than the gap between kernels:
  // 24^3 x 48 10.8 us with it, 9.8 without, 128^3 x 80 1132 and 1125 (32^3 x 80
  // alone 24.2 and 25.0).
  // stage: each warp copies the slots and gas records of its own cells and waits for
  // nothing else, so it must not read what another warp copies.  A warp of the last
  // block whose cells all lie past the end (its lanes would take the last cell's
  // record) copies nothing and leaves below; block barriers wait for the threads that
  // have not left.
  const bool alive = tile * CPB + warp * CW < a.n_cells;
  const int64_t kb = a.ptr[tile * CPB];
  const int64_t kc0 = a.ptr[c], kc1 = a.ptr[c + 1];
  {
    const int w0 = (int)(__shfl_sync(0xffffffffu, kc0, 0) - kb);
    const int w1 = (int)(__shfl_sync(0xffffffffu, kc1, 31) - kb);
    if (alive && !a.src_only) {
      const SlotF *g = (MOVING ? reinterpret_cast<const SlotF *>(a.slot) : a.slot_nb) + kb;
      for (int i = w0 + lane; i < w1; i += 32) {
        cp_async16(stage.slot + i, g + i);
        if (MOVING) cp_async4(stage.nbr + i, a.nbr + kb + i);
      }
    }
  }
  const int kind = a.kind[c];
  float2 NX[NQ], NY[NQ], NZ[NQ];
#pragma unroll
  for (int i = 0; i < NQ; ++i) {
    const float4 d = __ldg(qd.xy + sub + KT * i);
    const float2 z = __ldg(reinterpret_cast<const float2 *>(qd.zw + sub + KT * i));
    NX[i] = make_float2(d.x, d.y);
    NY[i] = make_float2(d.z, d.w);
    NZ[i] = z;
  }
  const float4 *tdir = reinterpret_cast<const float4 *>(a.dir) + 2 * KT * NQ + sub;
  float tx = 0.0f, ty = 0.0f, tz = 0.0f;
  if (TAIL) {
    const float4 d = __ldg(tdir);
    tx = d.x;
    ty = d.y;
    tz = d.z;
  }
  if (!alive) return;  // (at the top of the kernel it costs registers: 64^3 x 48 3 % longer)
  if (SMALL) asm volatile("griddepcontrol.wait;" ::: "memory");
  {
    for (int i = lane; i < 6 * CW; i += 32) {
      const int cc = warp * CW + i / 6, k = i % 6;
      const int64_t gc = tile * CPB + cc;
      if (gc < a.n_cells) {
        if (k < 4)
          cp_async16(reinterpret_cast<char *>(&stage.gas->gs[cc]) + 16 * k,
                     reinterpret_cast<const char *>(a.gs + gc) + 16 * k);
        else
          cp_async16(reinterpret_cast<char *>(&stage.gas->gd[cc]) + 16 * (k - 4),
                     reinterpret_cast<const char *>(a.gd + gc) + 16 * (k - 4));
      }
    }
  }
  // one warp prefetches the tile one wave of blocks ahead into L2, so that its
  // gathers and its own stage find the rows there instead of waiting on HBM
  const int64_t pc0 = (tile + kAhead) * CPB;
  const bool ahead = warp == 1 && pc0 < a.n_cells && !a.src_only;
  const int64_t pc1 = pc0 + CPB < a.n_cells ? pc0 + CPB : a.n_cells;
  int64_t pk0 = 0, pk1 = 0;
  if (ahead && lane == 0) {
    const unsigned n = (unsigned)(pc1 - pc0);
    pk0 = a.ptr[pc0];
    pk1 = a.ptr[pc1];
    l2_prefetch(a.I_in + (size_t)pc0 * RS, n * RS * (unsigned)sizeof(float));
    l2_prefetch(a.gs + pc0, n * (unsigned)sizeof(GasStatic));
    l2_prefetch(a.gd + pc0, n * (unsigned)sizeof(GasDyn));
    l2_prefetch(a.cellv + 4 * pc0, n * 16);
  }
  const float dtv = a.dt_r * a.inv_vol[c];
  const float4 cv = *reinterpret_cast<const float4 *>(a.cellv + 4 * c);
  cp_async_wait_all();
  __syncwarp();  // the warp's stage has landed
  if (ahead && lane == 0 && pk1 > pk0)
    l2_prefetch((MOVING ? reinterpret_cast<const SlotF *>(a.slot) : a.slot_nb) + pk0,
                (unsigned)(pk1 - pk0) * (unsigned)sizeof(SlotF));

  // ---------------- transport, I* = I - dt/V sum_f u I_up
  float2 IA[NQ], IB[NQ], IT = bcast(0.0f);
  {
    const float *o = a.I_in + (size_t)c * RS;
#pragma unroll
    for (int i = 0; i < NQ; ++i) {
      const float4 t = reinterpret_cast<const float4 *>(o)[sub + KT * i];
      IA[i] = make_float2(t.x, t.y);
      IB[i] = make_float2(t.z, t.w);
    }
    if (TAIL) IT = reinterpret_cast<const float2 *>(o)[2 * KT * NQ + sub];
  }
  if (!a.src_only) {
    QuadSums<NQ> u;
    quad_faces<NQ, TAIL, MOVING, SMALL ? quad_chunk<NQ>() : 0>(
        stage.slot, stage.nbr, (int)(kc0 - kb), (int)(kc1 - kb), a.I_in, RS, sub, NX, NY, NZ, tx,
        ty, tz, IA, IB, IT, u);
    const float2 mdt = bcast(-dtv), pdt = bcast(dtv);
#pragma unroll
    for (int i = 0; i < NQ; ++i) {
      IA[i] = pfma(mdt, u.CA[i], IA[i]);
      IB[i] = pfma(pdt, u.CB[i], IB[i]);
    }
    IT = pfma(mdt, u.CT, IT);
    if constexpr (MOVING) {
      if (a.gcl_rate) {
        // geometric conservation law: times V^n / V^{n+1} (see rt_step64.cu)
        const float2 ratio = bcast(rcp(fmaf(dtv, (float)a.gcl_rate[c], 1.0f)));
#pragma unroll
        for (int i = 0; i < NQ; ++i) {
          IA[i] = pmul(IA[i], ratio);
          IB[i] = pmul(IB[i], ratio);
        }
        IT = pmul(IT, ratio);
      }
    }
  }

  // ---------------- phase A: Gamma = 1 -+ v.n / c (first order in v/c), w~ =
  // w / Gamma^2 (normalised by their sum), S_I = sum w~ Gamma^4 I* / (1 + x Gamma), S_G
  // = sum w~ Gamma / (1 + x Gamma), S_1 = sum w~ / (1 + x Gamma).  To all orders Gamma
  // = gamma G: the weights' normalisation cancels gamma^2, so gamma enters only per
  // cell (x -> gamma x, S_I -> gamma^4 S_I, S_G -> gamma S_G and, in phase C, q ->
  // q / gamma^3; emitters: rate gamma, source / gamma^4).  A uniform weight cancels too.
  const float icr = a.inv_c_r;
  const float vx = cv.x * icr, vy = cv.y * icr, vz = cv.z * icr, eint = cv.w;
  const int li = (int)(c - tile * CPB);
  const GasStatic &gs = stage.gas->gs[li];
  float xs = a.dt_cbar_r * (gs.frkJ + gs.frkS);
  double2 ax = make_double2(0.0, 0.0);
  if (kind != RT_CELL_INTERIOR) ax = a.aux[c];
  if (kind == RT_CELL_EMITTER) xs = (float)(a.dt * a.cbar * ax.x);
  const float gam = frame_gamma(a.boost, vx, vy, vz);
  if (a.boost) xs *= gam;
  const bool uw = a.w_uniform;
  const float2 *W2 = reinterpret_cast<const float2 *>(a.wt2) + 2 * KT * NQ + sub;  // the tail pair's
  // the sums over a thread's angles run over its pairs in order, the first
  // angles' (x) and the antipodes' (y) apart
  float2 sIv = bcast(0.0f), sGv = sIv, s1v = sIv;
  {
    const float2 XS = bcast(xs), one = bcast(1.0f), m1 = bcast(-1.0f);
    const float2 VX = bcast(vx), VY = bcast(vy), VZ = bcast(vz);
#pragma unroll
    for (int i = 0; i < NQ; ++i) {
      const float2 BN = pfma(VX, NX[i], pfma(VY, NY[i], pmul(VZ, NZ[i])));
      const float2 GA = pfma(BN, m1, one), GB = padd(BN, one);
      const float2 GA2 = pmul(GA, GA), GB2 = pmul(GB, GB);
      // t = w / (Gamma^2 (1 + x Gamma)): one reciprocal per angle
      float2 ta = prcpf(pmul(GA2, pfma(XS, GA, one))), tb = prcpf(pmul(GB2, pfma(XS, GB, one)));
      float2 wa = bcast(a.w_uni), wb = wa;
      if (!uw) {
        const float4 d = __ldg(qd.zw + sub + KT * i);
        wa = make_float2(d.z, d.w);
        wb = __ldg(qd.wb + sub + KT * i);
      }
      ta = pmul(wa, ta);
      tb = pmul(wb, tb);
      const float2 ua = pmul(ta, pmul(GA2, GA2)), ub = pmul(tb, pmul(GB2, GB2));
      s1v.x = (s1v.x + ta.x) + ta.y;
      s1v.y = (s1v.y + tb.x) + tb.y;
      sIv.x = fmaf(ua.y, IA[i].y, fmaf(ua.x, IA[i].x, sIv.x));
      sIv.y = fmaf(ub.y, IB[i].y, fmaf(ub.x, IB[i].x, sIv.y));
      sGv.x = fmaf(ta.y, GA.y, fmaf(ta.x, GA.x, sGv.x));
      sGv.y = fmaf(tb.y, GB.y, fmaf(tb.x, GB.x, sGv.y));
    }
    if (TAIL) {
      const float bn = fmaf(vx, tx, fmaf(vy, ty, vz * tz));
      const float2 G = make_float2(1.0f - bn, 1.0f + bn), G2 = pmul(G, G);
      const float2 w = uw ? bcast(a.w_uni) : __ldg(W2);
      const float2 t = pmul(w, prcpf(pmul(G2, pfma(XS, G, one))));
      s1v = padd(s1v, t);
      sIv = pfma(pmul(t, pmul(G2, G2)), IT, sIv);
      sGv = pfma(t, G, sGv);
    }
  }
  float sI = cell_sum(sIv.x + sIv.y), sG = cell_sum(sGv.x + sGv.y), s1 = cell_sum(s1v.x + s1v.y);
  if (a.boost) {
    const float g2 = gam * gam;
    sI *= g2 * g2;
    sG *= gam;
  }

  // ---------------- phase B: the temperature equation, in every lane of the cell
  float q = 0.0f;  // dt cbar rho (kP B + kS J~)
  unsigned bad = 0;
  if (REFINE && a.beta_P_f != 0.0f) {
    // power-law opacities: the double Newton step takes a double power, so one
    // lane per cell runs it, between two block barriers
    if (sub == 0) {
      sh.sum[0][lc] = sI;
      sh.sum[1][lc] = sG;
      sh.sum[2][lc] = s1;
      sh.sum[3][lc] = eint;
    }
    __syncthreads();
    const int64_t cl = tile * CPB + lane;
    if (warp == cell_warp(tile, a.n_cells) && cl < a.n_cells) {
      float2 r = bcast(0.0f);
      if (a.kind[cl] == RT_CELL_INTERIOR) {
        float ql = 0.0f;
        unsigned bl = 0;
        // its coefficient check; the root itself is source_q_slow's
        if (!source_q_fast<REFINE>(a, stage.gas->gs[lane], sh.sum[0][lane], sh.sum[1][lane],
                                   sh.sum[2][lane], sh.sum[3][lane], ql, bl))
          r = source_q_slow(a, stage.gas->gs[lane], stage.gas->gd[lane], sh.sum[0][lane],
                            sh.sum[1][lane], sh.sum[2][lane], sh.sum[3][lane]);
        else
          r = make_float2(ql, __uint_as_float(bl));
      }
      sh.q[lane] = r.x;
      sh.bad[lane] = __float_as_uint(r.y);
    }
    __syncthreads();
    q = sh.q[lc];
    bad = sh.bad[lc];
    __syncthreads();  // before sh.sum and sh.bad are written again
  } else if (kind == RT_CELL_INTERIOR) {
    if (!source_q_fast<REFINE>(a, gs, sI, sG, s1, eint, q, bad)) {
      const GasDyn &gd = stage.gas->gd[li];
      const float2 r = REFINE || NQ > 2 ? source_q_slow(a, gs, gd, sI, sG, s1, eint)
                                        : source_q_double(a, gs, gd, sI, sG, s1, eint);
      q = r.x;
      bad |= __float_as_uint(r.y);
    }
  }

  // ---------------- phase C: interior I' = (I* Gamma^3 + q) / (Gamma^3 (1 + x Gamma));
  // emitter the same with x -> dt cbar (rho kappa)_src and q -> that rate times
  // I_src (Sec. 2.5); boundary I' = I* - f (I* - I0).  The gas receives the
  // difference of the stored intensities: the energy bookkeeping is then exact
  // in float.
  float dea = 0.0f, deb = 0.0f, dfx = 0.0f, dfy = 0.0f, dfz = 0.0f;
  {
    const bool bnd = kind == RT_CELL_BOUNDARY;
    float2 mf = bcast(0.0f);
    const float *I0 = a.I0;
    if (bnd) {
      mf = bcast(-(float)((ax.x <= a.dt) ? 1.0 : a.dt / ax.x));
      I0 = a.I0 + (size_t)a.bc_row[c] * RS;
    } else {
      if (kind == RT_CELL_EMITTER) q = xs * (float)ax.y;
      if (a.boost) q /= kind == RT_CELL_EMITTER ? (gam * gam) * (gam * gam) : gam * gam * gam;
    }
    const float2 QQ = bcast(q), XS = bcast(xs), one = bcast(1.0f), m1 = bcast(-1.0f);
    float *out = a.I_out + (size_t)c * RS;
#pragma unroll
    for (int i = 0; i < NQ; ++i) {
      const float4 xy = load_again(qd.xy + sub + KT * i), zw = load_again(qd.zw + sub + KT * i);
      float2 na, nb;
      if (bnd) {
        const float4 t = reinterpret_cast<const float4 *>(I0)[sub + KT * i];
        na = pfma(mf, psub(IA[i], make_float2(t.x, t.y)), IA[i]);
        nb = pfma(mf, psub(IB[i], make_float2(t.z, t.w)), IB[i]);
      } else {
        const float2 BN = pfma(bcast(vx), make_float2(xy.x, xy.y),
                               pfma(bcast(vy), make_float2(xy.z, xy.w),
                                    pmul(bcast(vz), make_float2(zw.x, zw.y))));
        const float2 GA = pfma(BN, m1, one), GB = padd(BN, one);
        const float2 GA3 = pmul(pmul(GA, GA), GA), GB3 = pmul(pmul(GB, GB), GB);
        na = pmul(pfma(IA[i], GA3, QQ), prcpf(pmul(GA3, pfma(XS, GA, one))));
        nb = pmul(pfma(IB[i], GB3, QQ), prcpf(pmul(GB3, pfma(XS, GB, one))));
      }
      if (live)
        reinterpret_cast<float4 *>(out)[sub + KT * i] = make_float4(na.x, na.y, nb.x, nb.y);
      float2 wa = bcast(a.w_uni), wb = wa;
      if (!uw) {
        wa = make_float2(zw.z, zw.w);
        wb = __ldg(qd.wb + sub + KT * i);
      }
      const float2 da = pmul(wa, psub(IA[i], na)), db = pmul(wb, psub(IB[i], nb));
      dea = (dea + da.x) + da.y;
      deb = (deb + db.x) + db.y;
      const float2 df = psub(da, db);  // the antipode has direction -n
      dfx = fmaf(xy.y, df.y, fmaf(xy.x, df.x, dfx));
      dfy = fmaf(xy.w, df.y, fmaf(xy.z, df.x, dfy));
      dfz = fmaf(zw.y, df.y, fmaf(zw.x, df.x, dfz));
    }
    if (TAIL) {
      const float4 n = load_again(tdir);
      float2 nt;
      if (bnd) {
        nt = pfma(mf, psub(IT, reinterpret_cast<const float2 *>(I0)[2 * KT * NQ + sub]), IT);
      } else {
        const float bn = fmaf(vx, n.x, fmaf(vy, n.y, vz * n.z));
        const float2 G = make_float2(1.0f - bn, 1.0f + bn);
        const float2 G3 = pmul(pmul(G, G), G);
        nt = pmul(pfma(IT, G3, QQ), prcpf(pmul(G3, pfma(XS, G, one))));
      }
      if (live) reinterpret_cast<float2 *>(out)[2 * KT * NQ + sub] = nt;
      const float2 w = uw ? bcast(a.w_uni) : __ldg(W2);
      const float2 d = pmul(w, psub(IT, nt));
      dea += d.x;
      deb += d.y;
      const float df = d.x - d.y;
      dfx = fmaf(n.x, df, dfx);
      dfy = fmaf(n.y, df, dfy);
      dfz = fmaf(n.z, df, dfz);
    }
  }
  if (SMALL) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  {
    const float v[4] = {dea + deb, dfx, dfy, dfz};
    cell_store4(v, sub, lc, sh.sum);
    if (sub == 0) sh.bad[lc] = bad;
  }
  __syncthreads();

  // ---------------- phase D: gas exchange, one lane per cell
  const int64_t cl = tile * CPB + lane;
  if (warp == cell_warp(tile, a.n_cells) && cl < a.n_cells) {
    unsigned b = sh.bad[lane];
    if (!isfinite(sh.sum[0][lane])) b |= ST_NONFINITE;
    gas_exchange<float, MOVING>(a, cl, stage.gas->gs[lane], stage.gas->gd[lane], sh.sum[0][lane],
                                sh.sum[1][lane], sh.sum[2][lane], sh.sum[3][lane], b);
  }
}

template <int NQ, bool TAIL, bool MOVING, bool SMALL>
cudaError_t launch_quad_as(rt_state *s, const StepArgs<float> &a, unsigned blocks) {
  const int cap = stage_cap(s->max_block_slots);
  const float4 *xy = reinterpret_cast<const float4 *>(s->d_qdir);
  const int Q = s->n_angles / 4;
  const QuadDir qd{xy, xy + Q, reinterpret_cast<const float2 *>(xy + 2 * Q)};
  auto *k = a.float_quartic ? quad_step_kernel<NQ, TAIL, MOVING, false, SMALL>
                            : quad_step_kernel<NQ, TAIL, MOVING, true, SMALL>;
  const cudaError_t e =
      launch_carved(k, blocks, NT, stage_bytes(cap, MOVING), quad_blocks<NQ, TAIL, SMALL>(),
                    sizeof(QuadShared), SMALL, s->stream, a, qd, cap);
  if (e != cudaSuccess) return e;
  s->launches++;
  return cudaGetLastError();
}

template <int NQ, bool TAIL, bool MOVING>
cudaError_t launch_quad(rt_state *s, double dt, const StepIO &io) {
  const StepArgs<float> a = step_args<float>(s, dt, io);
  const unsigned blocks = (unsigned)((s->n_cells + CPB - 1) / CPB);
  return blocks <= 2 * 152 ? launch_quad_as<NQ, TAIL, MOVING, true>(s, a, blocks)
                           : launch_quad_as<NQ, TAIL, MOVING, false>(s, a, blocks);
}

template <typename M, bool MOVING>
cudaError_t launch_pairs(rt_state *s, double dt, const StepIO &io) {
  const StepArgs<float> a = step_args<float>(s, dt, io);
  step_kernel<M, MOVING>
      <<<(unsigned)((s->n_cells + CPB - 1) / CPB), NT, 0, s->stream>>>(a);
  s->launches++;
  return cudaGetLastError();
}

template <bool MOVING, bool FULL>
cudaError_t dispatch_pairs(rt_state *s, double dt, const StepIO &io) {
  const int ppt = (s->n_angles / 2 + KT - 1) / KT;
  switch (ppt) {
    case 1: return launch_pairs<PairMap<float, 1, FULL>, MOVING>(s, dt, io);
    case 2: return launch_pairs<PairMap<float, 2, FULL>, MOVING>(s, dt, io);
    case 3: return launch_pairs<PairMap<float, 3, FULL>, MOVING>(s, dt, io);
    case 4: return launch_pairs<PairMap<float, 4, FULL>, MOVING>(s, dt, io);
    case 5: return launch_pairs<PairMap<float, 5, FULL>, MOVING>(s, dt, io);
    case 6: return launch_pairs<PairMap<float, 6, FULL>, MOVING>(s, dt, io);
    case 7: return launch_pairs<PairMap<float, 7, FULL>, MOVING>(s, dt, io);
    case 8: return launch_pairs<PairMap<float, 8, FULL>, MOVING>(s, dt, io);
    default: return cudaErrorInvalidValue;
  }
}

// Rows in the quad layout: A = 16 m (32 <= A <= 128), m / 2 quads per thread and a
// tail pair when m is odd.
template <bool MOVING> cudaError_t dispatch_quads(rt_state *s, double dt, const StepIO &io) {
  switch (s->n_angles / 16) {
    case 2: return launch_quad<1, false, MOVING>(s, dt, io);
    case 3: return launch_quad<1, true, MOVING>(s, dt, io);
    case 4: return launch_quad<2, false, MOVING>(s, dt, io);
    case 5: return launch_quad<2, true, MOVING>(s, dt, io);
    case 6: return launch_quad<3, false, MOVING>(s, dt, io);
    case 7: return launch_quad<3, true, MOVING>(s, dt, io);
    case 8: return launch_quad<4, false, MOVING>(s, dt, io);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t dispatch(rt_state *s, double dt, const StepIO &io) {
  if (s->quad_end > 0)  // rows in the quad layout
    return s->moving ? dispatch_quads<true>(s, dt, io) : dispatch_quads<false>(s, dt, io);
  if (cell_step_takes(s)) return launch_cell_step(s, dt, io);
  const bool full = (s->n_angles / 2) % KT == 0;
  if (s->moving)
    return full ? dispatch_pairs<true, true>(s, dt, io) : dispatch_pairs<true, false>(s, dt, io);
  return full ? dispatch_pairs<false, true>(s, dt, io) : dispatch_pairs<false, false>(s, dt, io);
}

}  // namespace

cudaError_t launch_step_io(rt_state *s, double dt, const StepIO &io) {
  return s->precision == RT_FP32 ? dispatch(s, dt, io) : launch_step_io64(s, dt, io);
}

cudaError_t launch_step(rt_state *s, double dt) {
  cudaError_t e;
  if (s->integrator == RT_VAN_LEER) {
    e = launch_step_vl(s, dt);
  } else if (s->n_groups > 1) {
    // frequency groups: the transport of all groups' intensities and the
    // coupled source step (one fused launch where the layout allows it)
    e = launch_group_step(s, dt, s->d_I[s->cur], s->d_I[s->cur ^ 1]);
  } else {
    const StepIO io{s->d_I[s->cur], s->d_I[s->cur ^ 1], false, true};
    e = launch_step_io(s, dt, io);
  }
  if (e == cudaSuccess) s->cur ^= 1;
  return e;
}

}  // namespace rt
