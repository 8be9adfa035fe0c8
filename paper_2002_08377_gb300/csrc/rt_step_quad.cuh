// The float step over quad rows: KT threads per cell, thread `sub` owning the
// quads sub + KT i (i < NQ) of a row, each as two packed FP32 units: (p, p+1) and
// their antipodes.
#pragma once

#include <cuda_runtime.h>

#include "rt_internal.cuh"
#include "rt_step_args.cuh"

namespace rt {
namespace step {

// Faces whose rows are loaded before the first one's arithmetic: what the
// registers of the kernel's occupancy allow without spills in the loop.
template <int NQ, bool TAIL, bool MOVING> constexpr int quad_unroll() {
  return NQ == 1 ? 3 : (TAIL && NQ == 2) || (MOVING && NQ > 2) ? 1 : 2;
}
__device__ __forceinline__ float2 bcast(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 pmax0(float2 v) {
  return make_float2(fmaxf(v.x, 0.0f), fmaxf(v.y, 0.0f));
}
__device__ __forceinline__ float2 prcpf(float2 v) { return make_float2(rcp(v.x), rcp(v.y)); }

// The direction table of the quads, each array contiguous over them:
// (nx0, nx1, ny0, ny1), (nz0, nz1, wa0, wa1), (wb0, wb1).
struct QuadDir {
  const float4 *xy, *zw;
  const float2 *wb;
};
// Loads that the compiler does not merge with an earlier one: the directions
// are read again where they are needed rather than held (and spilled) in between.
__device__ __forceinline__ float4 load_again(const float4 *p) {
  float4 v;
  asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p));
  return v;
}

// The flux sums of a thread's units: per quad sum u I_up of (p, p+1) and
// -sum u' I_up of their antipodes, the tail pair's (sum u I_up, sum u' I_up).
template <int NQ> struct QuadSums {
  float2 CA[NQ], CB[NQ], CT;
};

// sum_f u I_up over the slots [k0, k1) of the thread's cell, in slot order.  u of
// an angle through a face is d = n . s (minus A w . n), of its antipode -d (minus
// A w . n); per face and unit max(u, 0) times the own value plus min(u, 0) times
// the neighbour's, one of the two zero, so the pair of FMAs rounds as the
// single product u I_up does.  min(u, 0) = u - max(u, 0) exactly.  (I_in is not
// __restrict__: its loads must stay behind the wait for the kernel that wrote it.)
// CHUNK > 0 (meshes that leave the SMs mostly idle): the rows of CHUNK faces are
// loaded before the first one's arithmetic, the last chunk filled up with its
// last face's loads.
template <int NQ, bool TAIL, bool MOVING, int CHUNK>
__device__ __forceinline__ void quad_faces(const SlotF *slot, const int32_t *nbr, int k0, int k1,
                                           const float *I_in, int RS, int sub,
                                           const float2 (&NX)[NQ], const float2 (&NY)[NQ],
                                           const float2 (&NZ)[NQ], float tx, float ty, float tz,
                                           const float2 (&OA)[NQ], const float2 (&OB)[NQ],
                                           float2 OT, QuadSums<NQ> &o) {
  const float2 m1 = bcast(-1.0f);
#pragma unroll
  for (int i = 0; i < NQ; ++i) o.CA[i] = o.CB[i] = bcast(0.0f);
  o.CT = bcast(0.0f);
  struct Face {
    float4 s, v[NQ];
    float2 vt;
  };
  auto load = [&](int k, Face &f) {
    f.s = *reinterpret_cast<const float4 *>(slot + k);
    const int nb = MOVING ? nbr[k] : __float_as_int(f.s.w);
    const float *row = I_in + (size_t)nb * RS;
    const float4 *q = reinterpret_cast<const float4 *>(row) + sub;
#pragma unroll
    for (int i = 0; i < NQ; ++i) f.v[i] = q[KT * i];
    f.vt = TAIL ? reinterpret_cast<const float2 *>(row)[2 * KT * NQ + sub] : bcast(0.0f);
  };
  auto add = [&](const Face &f) {
    const float4 s = f.s;
    const float2 SX = bcast(s.x), SY = bcast(s.y), SZ = bcast(s.z);
#pragma unroll
    for (int i = 0; i < NQ; ++i) {
      const float2 va = make_float2(f.v[i].x, f.v[i].y), vb = make_float2(f.v[i].z, f.v[i].w);
      const float2 D = pfma(NX[i], SX, pfma(NY[i], SY, pmul(NZ[i], SZ)));
      float2 U = D, E = D;  // u of the angles, -u of their antipodes
      if (MOVING) {
        U = pfma(bcast(s.w), m1, D);
        E = padd(D, bcast(s.w));
      }
      const float2 UP = pmax0(U), UM = pfma(UP, m1, U);
      const float2 EP = MOVING ? pmax0(E) : UP, EM = MOVING ? pfma(EP, m1, E) : UM;
      o.CA[i] = pfma(UP, OA[i], pfma(UM, va, o.CA[i]));
      o.CB[i] = pfma(EM, OB[i], pfma(EP, vb, o.CB[i]));
    }
    if (TAIL) {
      const float d = fmaf(tx, s.x, fmaf(ty, s.y, tz * s.z));
      const float ua = MOVING ? d - s.w : d, ub = MOVING ? -d - s.w : -d;
      const bool pa = ua > 0.0f, pb = MOVING ? ub > 0.0f : !pa;
      o.CT = pfma(make_float2(ua, ub), make_float2(pa ? OT.x : f.vt.x, pb ? OT.y : f.vt.y), o.CT);
    }
  };
  if constexpr (CHUNK > 0) {
    for (int k = k0; k < k1; k += CHUNK) {
      Face f[CHUNK];
#pragma unroll
      for (int j = 0; j < CHUNK; ++j) load(k + j < k1 ? k + j : k1 - 1, f[j]);
#pragma unroll
      for (int j = 0; j < CHUNK; ++j)
        if (k + j < k1) add(f[j]);
    }
  } else {
    constexpr int kUnroll = quad_unroll<NQ, TAIL, MOVING>();
#pragma unroll kUnroll
    for (int k = k0; k < k1; ++k) {
      Face f;
      load(k, f);
      add(f);
    }
  }
}

// The sums of v[0..3] over a cell's 8 threads, written to out[k][lc] (a halving
// exchange; each value in a fixed order).
__device__ __forceinline__ void cell_store4(const float (&v)[4], int sub, int lc,
                                            float (*out)[CPB]) {
  static_assert(KT == 8, "three exchanges");
  const bool hi = sub & 4, odd = sub & 2;
  float a = hi ? v[2] : v[0], b = hi ? v[3] : v[1];
  a += __shfl_xor_sync(0xffffffffu, hi ? v[0] : v[2], 4);
  b += __shfl_xor_sync(0xffffffffu, hi ? v[1] : v[3], 4);
  float c = odd ? b : a;
  c += __shfl_xor_sync(0xffffffffu, odd ? a : b, 2);
  c += __shfl_xor_sync(0xffffffffu, c, 1);
  if (!(sub & 1)) out[(hi ? 2 : 0) + (odd ? 1 : 0)][lc] = c;
}

}  // namespace step
}  // namespace rt
