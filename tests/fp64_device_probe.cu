// Applies the functions of fp64_device.cuh, and CUDA's own, to arrays (test_gpu_fp64_device.py).
#include "fp64_device.cuh"

namespace gsis {
__global__ void probe(int which, int n, const double *x, const double *y, double *own, double *ref) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  own[i] = which == 0 ? rcp_newton(x[i]) : which == 1 ? quotient(x[i], y[i]) : root(x[i]);
  ref[i] = which == 0 ? __drcp_rn(x[i]) : which == 1 ? __ddiv_rn(x[i], y[i]) : __dsqrt_rn(x[i]);
}

// own: the viscosity at x of a cell whose anchor was taken at y; ref: at y itself
__global__ void probe_viscosity(MuSeries series, double mu0, double omega, int n, const double *x, const double *y,
                                double *own, double *ref) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double v[3] = {0.0, 0.0, 0.0};
  auto power = [](double T, double e) { return pow(T, e); };
  ref[i] = viscosity(y[i], mu0, omega, series, v, power);
  own[i] = viscosity(x[i], mu0, omega, series, v, power);
}

template <typename Launch>
static int on_device(int n, const double *x, const double *y, double *own, double *ref, Launch launch) {
  double *d = nullptr;
  const size_t b = (size_t)n * sizeof(double);
  cudaError_t e = cudaMalloc(&d, 4 * b);
  if (e == cudaSuccess) e = cudaMemcpy(d, x, b, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(d + n, y, b, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    launch(d, d + n, d + 2 * (size_t)n, d + 3 * (size_t)n);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(own, d + 2 * (size_t)n, b, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(ref, d + 3 * (size_t)n, b, cudaMemcpyDeviceToHost);
  if (d) cudaFree(d);
  return (int)e;
}
}  // namespace gsis

// host arrays of n values; 0 or the CUDA error
extern "C" int fp64_probe(int which, int n, const double *x, const double *y, double *own, double *ref) {
  return gsis::on_device(n, x, y, own, ref, [&](const double *a, const double *b, double *o, double *r) {
    gsis::probe<<<(n + 255) / 256, 256>>>(which, n, a, b, o, r);
  });
}

extern "C" int fp64_probe_viscosity(double mu0, double omega, int n, const double *x, const double *y, double *own, double *ref) {
  const gsis::MuSeries series = gsis::viscosity_series(omega);
  return gsis::on_device(n, x, y, own, ref, [&](const double *a, const double *b, double *o, double *r) {
    gsis::probe_viscosity<<<(n + 255) / 256, 256>>>(series, mu0, omega, n, a, b, o, r);
  });
}
