// fp64_device.cuh -- FP64 arithmetic of the kinetic kernel and of both synthetic solves: reciprocal,
// quotient, square root and viscosity in fewer instructions of the pipe that bounds them (a warp-wide
// FP64 instruction holds an SM's FP64 pipe for 19 cycles).  tests/test_gpu_fp64_device.py holds each
// against CUDA's own function over its range.
#pragma once
#include <cuda_runtime.h>

#include "gsis_internal.h"

namespace gsis {
namespace {
__device__ __forceinline__ long long dbits(double x) { return __double_as_longlong(x); }

// 1 / x by two Newton-Raphson steps y += y (1 - x y) from the hardware's approximation of its leading
// bits, for 2^-1022 <= |x| < 2^1022: densities, diagonals and the limiter's denominators, which are normal
// on any physical state (0, subnormal and larger values do not give CUDA's infinity or 0 but NaN).
// The residual of the last step is exact to far below an ulp, so the result is rounded once.
__device__ __forceinline__ double rcp_newton(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  y = fma(y, fma(-x, y, 1.0), y);
  return fma(y, fma(-x, y, 1.0), y);
}

// a / b for 0 <= a <= b < 2^1022: the quotient with the Newton reciprocal, corrected by its exact
// remainder (Markstein); the plain division where the approximation would flush b
__device__ __forceinline__ double quotient(double a, double b) {
  if (dbits(b) < 0x0060000000000000LL) return a / b;
  const double y = rcp_newton(b), q = a * y;
  return fma(fma(-b, q, a), y, q);
}

// sqrt(x) by Goldschmidt's iteration from the hardware's approximation of 1 / sqrt(x), the last step from
// the exact remainder x - g^2 (Markstein); the plain function outside the range where every intermediate
// is normal
__device__ __forceinline__ double root(double x) {
  if ((unsigned long long)(dbits(x) - 0x1000000000000000LL) > 0x6000000000000000ULL - 0x1000000000000000ULL) return sqrt(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  double h = __longlong_as_double(dbits(y) - (1LL << 52)), g = x * y;  // y / 2
  const double r = fma(-g, h, 0.5);
  g = fma(g, r, g);
  h = fma(h, r, h);
  return fma(fma(-g, g, x), h, g);
}

// Viscosity mu0 T^omega about the cell's anchor v = (1 / T0, mu0 T0^omega in two words), 1 / T0 a float so
// that x = T / T0 - 1 is rounded once: inside the series' range the binomial series of (1 + x)^omega - 1
// takes twelve FP64 instructions where the power takes a logarithm and an exponential, and its error is
// that of the anchor's power and of the last rounding, as for the product before.  A cell whose
// temperature has left that range (at the first step 1 / T0 = 0) gets a new anchor by `power(T, e)`.
template <typename Power>
__device__ __forceinline__ double viscosity(double T, double mu0, double omega, const MuSeries &series, double *v, Power power) {
  double x = fma(T, v[0], -1.0), hi = v[1], lo = v[2];
  if ((dbits(x) & 0x7fffffffffffffffLL) >= series.range) {
    const double i0 = (double)(float)(1.0 / T), p = power(i0, -omega);
    hi = mu0 * p;
    lo = fma(mu0, p, -hi);
    x = fma(T, i0, -1.0);
    v[0] = i0;
    v[1] = hi;
    v[2] = lo;
    if ((dbits(x) & 0x7fffffffffffffffLL) >= series.range) {  // 1 / T is no float, or there is no range
      v[0] = 0.0;
      return mu0 * power(T, omega);
    }
  }
  double s = series.c[MACRO_MU_SERIES - 1];
#pragma unroll
  for (int n = MACRO_MU_SERIES - 2; n >= 0; --n) s = fma(s, x, series.c[n]);
  return hi + fma(hi, s * x, lo);
}
}  // namespace
}  // namespace gsis
