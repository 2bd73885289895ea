// Applies the functions of fp64_device.cuh, and CUDA's own, to arrays (test_gpu_fp64_device.py).
#include "fp64_device.cuh"

namespace gsis {
__global__ void probe(int which, int n, const double *x, const double *y, double *own, double *ref) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  own[i] = which == 0 ? rcp_newton(x[i]) : which == 1 ? quotient(x[i], y[i]) : root(x[i]);
  ref[i] = which == 0 ? __drcp_rn(x[i]) : which == 1 ? __ddiv_rn(x[i], y[i]) : __dsqrt_rn(x[i]);
}
}  // namespace gsis

// host arrays of n values; 0 or the CUDA error
extern "C" int fp64_probe(int which, int n, const double *x, const double *y, double *own, double *ref) {
  double *d = nullptr;
  const size_t b = (size_t)n * sizeof(double);
  cudaError_t e = cudaMalloc(&d, 4 * b);
  if (e == cudaSuccess) e = cudaMemcpy(d, x, b, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(d + n, y, b, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    gsis::probe<<<(n + 255) / 256, 256>>>(which, n, d, d + n, d + 2 * (size_t)n, d + 3 * (size_t)n);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(own, d + 2 * (size_t)n, b, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(ref, d + 3 * (size_t)n, b, cudaMemcpyDeviceToHost);
  if (d) cudaFree(d);
  return (int)e;
}
