// Test-only shim: evaluates the library's scalar device helpers (joining a double-float to a double, reciprocal square
// root, square root, quotient) on host-provided inputs. Built by tests/test_device_scalar_gpu.py; not part of the
// library.
#include <cuda_runtime.h>

#include "../../paper_1608_03004_gb300/csrc/rlb_device_math.cuh"

__global__ void scalar_kernel(int which, const double* a, const double* b, double* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  if (which == 0) out[i] = rlbdev::df_join((float)a[i], (float)b[i]);
  if (which == 1) out[i] = rlbdev::rsqrt_nr(a[i]);
  if (which == 2) out[i] = rlbdev::sqrt_nr(a[i]);
  if (which == 3) out[i] = rlbdev::div_nr(a[i], b[i]);
  if (which == 4) out[i] = rlbdev::df_split(a[i]).hi;
}

extern "C" int ds_eval(int which, const double* a, const double* b, double* out, int n) {
  double* d = nullptr;
  if (cudaMalloc(&d, 3 * (size_t)n * sizeof(double)) != cudaSuccess) return 1;
  cudaMemcpy(d, a, n * sizeof(double), cudaMemcpyHostToDevice);
  cudaMemcpy(d + n, b, n * sizeof(double), cudaMemcpyHostToDevice);
  scalar_kernel<<<(n + 255) / 256, 256>>>(which, d, d + n, d + 2 * n, n);
  const cudaError_t e = cudaMemcpy(out, d + 2 * n, n * sizeof(double), cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e == cudaSuccess ? 0 : 2;
}
