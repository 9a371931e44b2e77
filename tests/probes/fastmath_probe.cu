// Evaluates the kernels' own elementary functions on arrays, for
// test_gpu_fp64_rounding.py.
#include "../../paper_2003_09926_gb300/csrc/jz_fastmath.cuh"

using namespace jz::stg;

__global__ void k_eval(int which, int n, const double* x, double* y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  switch (which) {
    case 0: y[i] = rcp_d(x[i]); break;
    case 1: y[i] = sqrt_d(x[i]); break;
    case 2: y[i] = jm23_d(x[i]); break;
    default: {  // CUDA's cbrt, a product and a division
      const double c = cbrt(x[i]);
      y[i] = 1.0 / (c * c);
    }
  }
}

// n groups of five FP32 values (as doubles) widened to FP64
__global__ void k_widen(int n, const double* x, double* y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float f[5];
  for (int v = 0; v < 5; ++v) f[v] = (float)x[5 * i + v];
  double d[5];
  widen5(f, d);
  for (int v = 0; v < 5; ++v) y[5 * i + v] = d[v];
}

// y = f(x) for n host values; returns a CUDA error code
extern "C" int fastmath_eval(int which, int n, const double* x, double* y) {
  double* d = nullptr;
  cudaError_t e = cudaMalloc(&d, 2 * sizeof(double) * (size_t)n);
  if (e != cudaSuccess) return (int)e;
  e = cudaMemcpy(d, x, sizeof(double) * (size_t)n, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    if (which == 4)
      k_widen<<<(n / 5 + 255) / 256, 256>>>(n / 5, d, d + n);
    else
      k_eval<<<(n + 255) / 256, 256>>>(which, n, d, d + n);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(y, d + n, sizeof(double) * (size_t)n, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return (int)e;
}
