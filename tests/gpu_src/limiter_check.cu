// Test-only shim: the packed double-float limiter with a different interface in each half, and the adjoint's gradient
// of the interface value, on host-provided inputs. Built by tests/test_limiter_gpu.py; not part of the library.
#include <cuda_runtime.h>

#include "../../paper_1608_03004_gb300/csrc/rlb_device_math.cuh"

using namespace rlbdev;

// Interface values of two stencils at once, as the FP64 stage kernel forms them: v holds 5 samples of each (wind toward
// increasing index), out the two values.
__device__ void both(const double* v, const double* w, double* out) {
  DF2 D[4];
  for (int k = 0; k < 4; ++k) {
    const DF a = df_split(v[k + 1] - v[k]), b = df_split(w[k + 1] - w[k]);
    D[k] = {f2(a.hi, b.hi), f2(a.lo, b.lo)};
  }
  const DF e = df_split(3.0 * WENO_EPS);
  const F2 nz = minus_zero2();
  DF2 a[3], b[3], c[3];
  for (int k = 0; k < 3; ++k) weno5_pair_df2(D[k], D[k + 1], f2(-e.hi), f2(e.lo), nz, a[k], b[k], c[k]);
  const DF2 G = weno5_combine6_df2(a[0], b[1], c[2], D[0], D[1], D[2], D[3], nz);
  out[0] = fma(df_join(lo_of(G.hi), lo_of(G.lo)), 1.0 / 6.0, v[2]);
  out[1] = fma(df_join(hi_of(G.hi), hi_of(G.lo)), 1.0 / 6.0, w[2]);
}

__global__ void pair_kernel(const double* v, const double* w, double* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) both(v + 5 * i, w + 5 * i, out + 2 * i);
}

// out: dPhi/dv_m, m = 0..4, of the samples v
__global__ void grad_kernel(const double* v, const double*, double* out, int n) {
  __shared__ double cst[ADJ_CST];
  if (threadIdx.x < ADJ_CST) cst[threadIdx.x] = grad_constant(threadIdx.x);
  __syncthreads();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double* s = v + 5 * i;
  double g[4];
  weno5_grad(s[1] - s[0], s[2] - s[1], s[3] - s[2], s[4] - s[3], 3.0 * WENO_EPS, cst, g);
  for (int m = 0; m < 5; ++m)
    out[5 * i + m] = ((m > 0 ? g[m - 1] : 0.0) - (m < 4 ? g[m] : 0.0)) * (2.0 / 3.0) + (m == 2 ? 1.0 : 0.0);
}

extern "C" int lm_eval(int which, const double* v, const double* w, double* out, int n) {
  const int no = which == 0 ? 2 : 5;
  double *d = nullptr, *o = nullptr;
  if (cudaMalloc(&d, 10 * (size_t)n * sizeof(double)) != cudaSuccess) return 1;
  if (cudaMalloc(&o, no * (size_t)n * sizeof(double)) != cudaSuccess) return 1;
  cudaMemcpy(d, v, 5 * (size_t)n * sizeof(double), cudaMemcpyHostToDevice);
  cudaMemcpy(d + 5 * (size_t)n, w, 5 * (size_t)n * sizeof(double), cudaMemcpyHostToDevice);
  if (which == 0)
    pair_kernel<<<(n + 127) / 128, 128>>>(d, d + 5 * (size_t)n, o, n);
  else
    grad_kernel<<<(n + 127) / 128, 128>>>(d, d + 5 * (size_t)n, o, n);
  const cudaError_t e = cudaMemcpy(out, o, no * (size_t)n * sizeof(double), cudaMemcpyDeviceToHost);
  cudaFree(d);
  cudaFree(o);
  return e == cudaSuccess ? 0 : 2;
}
