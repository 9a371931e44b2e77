// Evaluates the FP64 stage kernel's face flux on arrays, for
// test_gpu_fp64_rounding.py.
#include "../../paper_2003_09926_gb300/csrc/jz_stage_d.cu"

namespace jz {
int device_sm_count() { return 152; }
void count_launches(uint64_t) {}
}  // namespace jz

// per face: Ga 7, Gb 7, qm 5, qa 5, qb 5, qp 5 -> twice the face flux 5
constexpr int IN = 34, OUT = 5;

__global__ void k_face(int n, double k2, double k4, const double* x, double* y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  jz::stg::KConst<double> c = {};
  c.k2 = k2;
  c.k4 = k4;
  const double* p = x + (size_t)i * IN;
  double h[OUT];
  jz::face_d(c, p, p + 7, p + 14, p + 19, p + 24, p + 29, h);
  for (int v = 0; v < OUT; ++v) y[(size_t)i * OUT + v] = h[v];
}

// returns a CUDA error code
extern "C" int face_eval(int n, double k2, double k4, const double* x, double* y) {
  double* d = nullptr;
  cudaError_t e = cudaMalloc(&d, sizeof(double) * (IN + OUT) * (size_t)n);
  if (e != cudaSuccess) return (int)e;
  e = cudaMemcpy(d, x, sizeof(double) * IN * (size_t)n, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    k_face<<<(n + 127) / 128, 128>>>(n, k2, k4, d, d + (size_t)n * IN);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(y, d + (size_t)n * IN, sizeof(double) * OUT * (size_t)n, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return (int)e;
}
