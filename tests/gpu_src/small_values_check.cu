// Test-only shim: the library's conversions and roots at values below the normal range, on host-provided inputs. Built
// by tests/test_small_values_gpu.py; not part of the library.
#include <cuda_runtime.h>

#include "../../paper_1608_03004_gb300/csrc/rlb_device_math.cuh"

__global__ void small_kernel(int which, const double* a, const double* b, double* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  if (which == 0) out[i] = (double)rlbdev::round_f32(a[i]);
  if (which == 1) out[i] = rlbdev::df_sum((float)a[i], (float)b[i]);
  if (which == 2) out[i] = rlbdev::sqrt_nr(a[i]);
}

extern "C" int sv_eval(int which, const double* a, const double* b, double* out, int n) {
  double* d = nullptr;
  if (cudaMalloc(&d, 3 * (size_t)n * sizeof(double)) != cudaSuccess) return 1;
  cudaMemcpy(d, a, n * sizeof(double), cudaMemcpyHostToDevice);
  cudaMemcpy(d + n, b, n * sizeof(double), cudaMemcpyHostToDevice);
  small_kernel<<<(n + 255) / 256, 256>>>(which, d, d + n, d + 2 * n, n);
  const cudaError_t e = cudaMemcpy(out, d + 2 * n, n * sizeof(double), cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e == cudaSuccess ? 0 : 2;
}
