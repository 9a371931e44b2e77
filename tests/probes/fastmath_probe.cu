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
    default: y[i] = Fn<double>::jm23(x[i]); break;  // CUDA's cbrt, a product and a division
  }
}

// y = f(x) for n host values; returns a CUDA error code
extern "C" int fastmath_eval(int which, int n, const double* x, double* y) {
  double* d = nullptr;
  cudaError_t e = cudaMalloc(&d, 2 * sizeof(double) * (size_t)n);
  if (e != cudaSuccess) return (int)e;
  e = cudaMemcpy(d, x, sizeof(double) * (size_t)n, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    k_eval<<<(n + 255) / 256, 256>>>(which, n, d, d + n);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(y, d + n, sizeof(double) * (size_t)n, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return (int)e;
}
