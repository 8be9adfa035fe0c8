// refine_quartic beside refine_root on the same equations (test_gpu_refine.py).
#include "rt_step_source.cuh"

__global__ void probe_kernel(const float *alpha, const double *beta, const float *g, const float *T0,
                             int64_t n, float *quick, uint8_t *took, float *full) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float T = 0.0f;
  took[i] = rt::step::refine_quartic(alpha[i], beta[i], (float)beta[i], g[i], T0[i], &T);
  quick[i] = T;
  full[i] = (float)rt::step::refine_root(alpha[i], 0.0f, 0.0, beta[i], g[i], T0[i]);
}

// the float Newton's root of alpha T^4 + beta T = g from T (in place)
__global__ void root_kernel(const float *alpha, const double *beta, const float *g, int64_t n,
                            float tol, float *T) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float r = 0.0f;
  rt::step::quartic_root(alpha[i], (float)beta[i], g[i], T[i], tol, 64, &r);
  T[i] = r;
}

extern "C" int probe(const float *alpha, const double *beta, const float *g, float *T0, int64_t n,
                     float tol, float *quick, uint8_t *took, float *full) {
  const unsigned blocks = (unsigned)((n + 255) / 256);
  if (tol > 0.0f) root_kernel<<<blocks, 256>>>(alpha, beta, g, n, tol, T0);
  probe_kernel<<<blocks, 256>>>(alpha, beta, g, T0, n, quick, took, full);
  return (int)cudaDeviceSynchronize();
}
