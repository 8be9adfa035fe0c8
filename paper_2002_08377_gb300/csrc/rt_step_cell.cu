// The fused radiation step of float states with at most 8 angles (S2), rows in the
// pair layout, two threads per cell.
//
// The tile kernel's 8 threads per cell leave half its lanes idle here (4 pairs of
// 8 angles) and repeat every per-cell and per-face operation in 8 lanes for little
// arithmetic.  Thread t of a cell holds the pairs 2t, 2t + 1: one 16-byte load per
// face, a neighbour's 32-byte row in one L1 wavefront (one thread per cell took
// four: 97 us at 64^3).  The sums are taken in the tile kernel's order ((s0 + s2) +
// (s1 + s3)), so both give the same bits.  The block's face slots are staged in
// shared memory; the double gas update runs after the block's second barrier with
// all lanes of two warps, one lane per cell.  The directions and weights come with
// the kernel arguments (constant bank).
#include <cuda_runtime.h>

#include "rt_internal.cuh"
#include "rt_step_args.cuh"
#include "rt_step_source.cuh"

namespace rt {
namespace {
using namespace step;

constexpr int kCells = 64;  // cells per block
constexpr int kThreads = 2 * kCells;

struct SmallSet {  // pair 2t + j of thread t at [t][j] (zero weights: no such pair)
  float x[2][2], y[2][2], z[2][2], wa[2][2], wb[2][2];
};

// The sum over a cell's pairs from the thread's two partial sums, in both threads.
__device__ __forceinline__ float pair_tree(float s0, float s1) {
  const float w0 = s0 + __shfl_xor_sync(0xffffffffu, s0, 1);
  const float w1 = s1 + __shfl_xor_sync(0xffffffffu, s1, 1);
  return w0 + w1;
}

template <bool MOVING>
__global__ void __launch_bounds__(kThreads, 8)
    cell_step_kernel(const __grid_constant__ StepArgs<float> a,
                     const __grid_constant__ SmallSet set, int cap) {
  extern __shared__ __align__(16) unsigned char cell_dyn[];
  __shared__ float sum[4][kCells];
  __shared__ unsigned bad_s[kCells];
  SlotF *slot = reinterpret_cast<SlotF *>(cell_dyn);
  int32_t *nbr = reinterpret_cast<int32_t *>(slot + cap);
  const int64_t c0 = (int64_t)blockIdx.x * kCells;
  const int lc = threadIdx.x / 2, t = threadIdx.x % 2;
  const int64_t cend = c0 + kCells < a.n_cells ? c0 + kCells : a.n_cells;
  const bool live = c0 + lc < a.n_cells;
  const int64_t c = live ? c0 + lc : a.n_cells - 1;  // dead lanes shadow the last cell
  const int64_t kb = a.ptr[c0];
  const int cnt = (int)(a.ptr[cend] - kb);
  if (!a.src_only) {
    const SlotF *g = (MOVING ? reinterpret_cast<const SlotF *>(a.slot) : a.slot_nb) + kb;
    for (int i = threadIdx.x; i < cnt; i += kThreads) {
      cp_async16(slot + i, g + i);
      if (MOVING) cp_async4(nbr + i, a.nbr + kb + i);
    }
  }
  const int H = a.half, RS = a.row;
  const bool has0 = 2 * t < H, has1 = 2 * t + 1 < H;
  const bool whole = H == 4;  // 16-byte accesses: both pairs there, rows 32 bytes apart
  float nx[2], ny[2], nz[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    nx[j] = t ? set.x[1][j] : set.x[0][j];
    ny[j] = t ? set.y[1][j] : set.y[0][j];
    nz[j] = t ? set.z[1][j] : set.z[0][j];
  }
  auto load = [&](const float *row) {
    float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (whole) {
      v = reinterpret_cast<const float4 *>(row)[t];
    } else {
      const float2 *p = reinterpret_cast<const float2 *>(row) + 2 * t;
      if (has0) {
        const float2 x = p[0];
        v.x = x.x;
        v.y = x.y;
      }
      if (has1) {
        const float2 x = p[1];
        v.z = x.x;
        v.w = x.y;
      }
    }
    return v;
  };
  float4 I = load(a.I_in + (size_t)c * RS);  // (I_p, I_p', I_p+1, I_p+1')
  cp_async_wait_all();
  __syncthreads();

  // ---------------- transport, I* = I - dt/V sum_f u I_up, faces in slot order
  if (!a.src_only) {
    float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    const int k0 = (int)(a.ptr[c] - kb), k1 = (int)(a.ptr[c + 1] - kb);
#pragma unroll 4
    for (int k = k0; k < k1; ++k) {
      const float4 s = *reinterpret_cast<const float4 *>(slot + k);
      const int nb = MOVING ? nbr[k] : __float_as_int(s.w);
      const SlotF sl{s.x, s.y, s.z, s.w};
      const float w = MOVING ? s.w : 0.0f;
      const float4 v = load(a.I_in + (size_t)nb * RS);
      face_pair<float, MOVING>(slot_dot(nx[0], ny[0], nz[0], sl), w, v.x, v.y, I.x, I.y, acc.x,
                               acc.y);
      face_pair<float, MOVING>(slot_dot(nx[1], ny[1], nz[1], sl), w, v.z, v.w, I.z, I.w, acc.z,
                               acc.w);
    }
    const float dtv = a.dt_r * a.inv_vol[c];
    I = make_float4(fmaf(-dtv, acc.x, I.x), fmaf(-dtv, acc.y, I.y), fmaf(-dtv, acc.z, I.z),
                    fmaf(-dtv, acc.w, I.w));
    if (MOVING && a.gcl_rate) {
      const float ratio = rcp(fmaf(dtv, (float)a.gcl_rate[c], 1.0f));
      I = make_float4(I.x * ratio, I.y * ratio, I.z * ratio, I.w * ratio);
    }
  }

  // ---------------- phase A (see rt_step.cu)
  const int kind = a.kind[c];
  const float4 cv = *reinterpret_cast<const float4 *>(a.cellv + 4 * c);
  const float icr = a.inv_c_r;
  const float vx = cv.x * icr, vy = cv.y * icr, vz = cv.z * icr;
  const GasStatic &gs = a.gs[c];
  float xs = a.dt_cbar_r * (gs.frkJ + gs.frkS);
  const float gam = frame_gamma(a.boost, vx, vy, vz);
  if (a.boost) xs *= gam;
  const float2 one = make_float2(1.0f, 1.0f);
  float2 Iv[2] = {make_float2(I.x, I.y), make_float2(I.z, I.w)}, w[2], G[2];
  float pI[2], pG[2], p1[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    w[j] = t ? make_float2(set.wa[1][j], set.wb[1][j]) : make_float2(set.wa[0][j], set.wb[0][j]);
    const float bn = fmaf(vx, nx[j], fmaf(vy, ny[j], vz * nz[j]));
    G[j] = make_float2(1.0f - bn, 1.0f + bn);
    const float2 G2 = pmul(G[j], G[j]);
    const float2 q = pmul(w[j], prcp<float>(pmul(G2, pfma(make_float2(xs, xs), G[j], one))));
    const float2 u = pmul(pmul(q, pmul(G2, G2)), Iv[j]), g = pmul(q, G[j]);
    p1[j] = q.x + q.y;
    pI[j] = u.x + u.y;
    pG[j] = g.x + g.y;
  }
  float sI = pair_tree(pI[0], pI[1]), sG = pair_tree(pG[0], pG[1]);
  const float s1 = pair_tree(p1[0], p1[1]);
  if (a.boost) {
    const float g2 = gam * gam;
    sI *= g2 * g2;
    sG *= gam;
  }

  // ---------------- phase B, in both threads
  float q = 0.0f;
  unsigned bad = 0;
  if (kind == RT_CELL_INTERIOR) {
    const bool ok = a.float_quartic ? source_q_fast<false>(a, gs, sI, sG, s1, cv.w, q, bad)
                                    : source_q_fast<true>(a, gs, sI, sG, s1, cv.w, q, bad);
    if (!ok) {
      const float2 r = source_q_slow(a, gs, a.gd[c], sI, sG, s1, cv.w);
      q = r.x;
      bad |= __float_as_uint(r.y);
    }
  }

  // ---------------- phase C
  float f = 0.0f;
  float4 i0 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  if (kind == RT_CELL_BOUNDARY) {
    const double2 ax = a.aux[c];
    f = (float)((ax.x <= a.dt) ? 1.0 : a.dt / ax.x);
    i0 = load(a.I0 + (size_t)a.bc_row[c] * RS);
  } else if (kind == RT_CELL_EMITTER) {
    const double2 ax = a.aux[c];
    xs = (float)(a.dt * a.cbar * ax.x);
    if (a.boost) xs *= gam;
    q = xs * (float)ax.y;
    if (a.boost) q /= (gam * gam) * (gam * gam);
  } else if (a.boost) {
    q /= gam * gam * gam;
  }
  float2 n[2];
  float pe[2], px[2], py[2], pz[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    if (kind == RT_CELL_BOUNDARY) {
      const float2 b = j ? make_float2(i0.z, i0.w) : make_float2(i0.x, i0.y);
      n[j] = pfma(make_float2(-f, -f), psub(Iv[j], b), Iv[j]);
    } else {
      const float2 G3 = pmul(pmul(G[j], G[j]), G[j]);
      n[j] = pmul(pfma(Iv[j], G3, make_float2(q, q)),
                  prcp<float>(pmul(G3, pfma(make_float2(xs, xs), G[j], one))));
    }
    const float2 d = pmul(w[j], psub(Iv[j], n[j]));
    const float df = d.x - d.y;  // the antipode has direction -n
    pe[j] = d.x + d.y;
    px[j] = nx[j] * df;
    py[j] = ny[j] * df;
    pz[j] = nz[j] * df;
  }
  if (live) {
    float *row = a.I_out + (size_t)c * RS;
    if (whole) {
      reinterpret_cast<float4 *>(row)[t] = make_float4(n[0].x, n[0].y, n[1].x, n[1].y);
    } else {
      if (has0) reinterpret_cast<float2 *>(row)[2 * t] = n[0];
      if (has1) reinterpret_cast<float2 *>(row)[2 * t + 1] = n[1];
    }
  }
  const float v[4] = {pair_tree(pe[0], pe[1]), pair_tree(px[0], px[1]), pair_tree(py[0], py[1]),
                      pair_tree(pz[0], pz[1])};
  if (!t) {
#pragma unroll
    for (int k = 0; k < 4; ++k) sum[k][lc] = v[k];
    bad_s[lc] = bad;
  }
  __syncthreads();

  // ---------------- phase D: gas exchange, one lane per cell
  const int64_t cl = c0 + threadIdx.x;
  if (threadIdx.x < kCells && cl < a.n_cells) {
    unsigned b = bad_s[threadIdx.x];
    const float de = sum[0][threadIdx.x];
    if (!isfinite(de)) b |= ST_NONFINITE;
    gas_exchange<float, MOVING>(a, cl, a.gs[cl], a.gd[cl], de, sum[1][threadIdx.x],
                                sum[2][threadIdx.x], sum[3][threadIdx.x], b);
  }
}

}  // namespace

bool cell_step_takes(const rt_state *s) {
  // at every mesh size (us per step with 8 angles, tile kernel and this one: 12^3
  // 7.8 and 6.3, 24^3 8.6 and 7.0, 32^3 15.4 and 9.0, 40^3 28.5 and 12.7, 64^3 131
  // and 47); with 24 angles the tile kernel's wider row loads win (64^3 133, one
  // thread per cell 153)
  return s->precision == RT_FP32 && s->quad_end == 0 && s->n_angles <= 8 &&
         s->max_block_slots <= STAGE_SLOTS;
}

cudaError_t launch_cell_step(rt_state *s, double dt, const StepIO &io) {
  static_assert(kCells == 2 * CPB, "the stage holds two tiles' slots");
  const StepArgs<float> a = step_args<float>(s, dt, io);
  SmallSet d{};
  for (int p = 0; p < s->n_angles / 2; ++p) {
    d.x[p / 2][p % 2] = s->small_dir[3 * p];
    d.y[p / 2][p % 2] = s->small_dir[3 * p + 1];
    d.z[p / 2][p % 2] = s->small_dir[3 * p + 2];
    d.wa[p / 2][p % 2] = s->small_w[2 * p];
    d.wb[p / 2][p % 2] = s->small_w[2 * p + 1];
  }
  const int cap = (int)((2 * s->max_block_slots + 7) & ~int64_t(7));
  const unsigned blocks = (unsigned)((s->n_cells + kCells - 1) / kCells);
  const size_t sm = (size_t)cap * (sizeof(SlotF) + (s->moving ? sizeof(int32_t) : 0));
  auto *k = s->moving ? cell_step_kernel<true> : cell_step_kernel<false>;
  const cudaError_t e =
      launch_carved(k, blocks, kThreads, sm, 8, 5 * kCells * sizeof(float), false, s->stream, a, d,
                    cap);
  if (e != cudaSuccess) return e;
  s->launches++;
  return cudaGetLastError();
}

}  // namespace rt
