// kinetic_device.cuh -- device helpers shared by the kinetic kernels: storage of the VDF and its
// lazy correction, the reference distributions, comparisons, the limiter, warp reductions.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <type_traits>

#include "fp64_device.cuh"
#include "gsis_internal.h"

namespace gsis {

// VDF element load / store between the storage type S and the arithmetic type T: plain for
// S = T; BF16 storage widens exactly to FP32 on load and rounds to nearest even on store.
template <typename T, typename S>
struct Fio {
  static __device__ __forceinline__ T ld(const S *p) { return *p; }
  static __device__ __forceinline__ void st(S *p, T v) { *p = v; }
};
template <>
struct Fio<float, __nv_bfloat16> {
  static __device__ __forceinline__ float ld(const __nv_bfloat16 *p) { return __bfloat162float(*p); }
  static __device__ __forceinline__ void st(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }
};

__device__ __forceinline__ float dexp(float x) { return __expf(x); }
__device__ __forceinline__ double dexp(double x) { return exp(x); }
__device__ __forceinline__ float ddiv(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double ddiv(double a, double b) { return a / b; }

// Wall Maxwellian M(xi; u_w, T_w) with unit density, in the arithmetic type (an FP64 pow per
// lane would cost FP64-rate time on this GPU in every CTA's set-up)
template <typename T>
__device__ __forceinline__ T wall_maxwellian(const double *uT, T x, T y, T z) {
  const T ux = (T)uT[0], uy = (T)uT[1], uz = (T)uT[2], Tw = (T)uT[3];
  const T cx = x - ux, cy = y - uy, cz = z - uz;
  const T pT = (T)3.14159265358979323846 * Tw;
  const T norm = (T)1 / (pT * sqrt(pT));  // (pi T_w)^(-3/2)
  return norm * dexp(-(cx * cx + cy * cy + cz * cz) / Tw);
}

// f^n = s f_raw + Cn M(un, Tn) - Co M(uo, To)   (Eq. updatef applied on load)
template <typename T>
__device__ __forceinline__ T corrected(T fraw, const T *st, T x, T y, T z) {
  T cx = x - st[0], cy = y - st[1], cz = z - st[2];
  T mn = st[4] * dexp(-(cx * cx + cy * cy + cz * cz) * st[3]);
  cx = x - st[5]; cy = y - st[6]; cz = z - st[7];
  T mo = st[9] * dexp(-(cx * cx + cy * cy + cz * cz) * st[8]);
  return st[10] * fraw + mn - mo;
}

// BF16 and FP32 storage keep f_raw relative to a per-cell Maxwellian, the Maxwellian of W^n of
// the kinetic step that stored it (state values 16..20): the stored deviation is small next to
// f, and so is its round-off.  FP64 stores f_raw itself (an FP64 exponential per point costs
// more than its round-off is worth).
template <typename S>
struct StoredRelative : std::false_type {};
template <>
struct StoredRelative<__nv_bfloat16> : std::true_type {};
template <>
struct StoredRelative<float> : std::true_type {};

// state values a loader of stored f needs: 24 with the storage reference (FP32, BF16), 12 for
// FP64 storage (slots 0..10, rounded up to whole 16-byte rows)
template <typename S>
__host__ __device__ constexpr int state_len() { return StoredRelative<S>::value ? 24 : 12; }

// f^n from a stored value: f_raw = stored (+ M_r for relative storage), then Eq. updatef
template <typename T, typename S>
__device__ __forceinline__ T corrected_stored(T stored, const T *st, T x, T y, T z) {
  if constexpr (StoredRelative<S>::value) {
    const T cx = x - st[16], cy = y - st[17], cz = z - st[18];
    stored += st[20] * dexp(-(cx * cx + cy * cy + cz * cz) * st[19]);
  }
  return corrected(stored, st, x, y, z);
}

// f^n of the NV reduced VDFs from their stored values, sharing the Maxwellians: f0 as above;
// f1 (Rykov) carries the internal-energy factor d_r T_r / 4 of each Maxwellian (state values
// 21, 29, 39), in its storage reference and in Eq. updatef alike.
template <typename T, typename S, int NV>
__device__ __forceinline__ void corrected_all(const T *stored, const T *st, T x, T y, T z, T *f) {
  T cx = x - st[0], cy = y - st[1], cz = z - st[2];
  const T mn = st[4] * dexp(-(cx * cx + cy * cy + cz * cz) * st[3]);
  cx = x - st[5]; cy = y - st[6]; cz = z - st[7];
  const T mo = st[9] * dexp(-(cx * cx + cy * cy + cz * cz) * st[8]);
  T raw[NV];
#pragma unroll
  for (int q = 0; q < NV; ++q) raw[q] = stored[q];
  if constexpr (StoredRelative<S>::value) {
    cx = x - st[16]; cy = y - st[17]; cz = z - st[18];
    const T mr = st[20] * dexp(-(cx * cx + cy * cy + cz * cz) * st[19]);
    raw[0] += mr;
    if constexpr (NV == 2) raw[1] += st[21] * mr;
  }
  f[0] = st[10] * raw[0] + mn - mo;
  if constexpr (NV == 2) f[1] = st[10] * raw[1] + st[29] * mn - st[39] * mo;
}

// Reference distributions of the state W^n (Section 2.2), c = xi - u_n, c2 = |c|^2:
//   Shakhov: g0 = M_t [1 + A q_t.c (c^2/T_t - 5/2)];
//   Rykov:   g_q = (1 - 1/Z_r) g_qt + g_qr / Z_r with the translational (T_t) and equilibrium
//            (T) Maxwellians, heat fluxes q0, q1 and the internal-energy factors (state 24..38).
// mw returns M_t, the Maxwellian relative storage refers to.
template <typename T, int NV>
__device__ __forceinline__ void reference(const T *st, T cx, T cy, T cz, T c2, T &mw, T *g) {
  const T et = dexp(-c2 * st[3]);
  mw = st[4] * et;
  const T g0t = mw * ((T)1 + (st[12] * cx + st[13] * cy + st[14] * cz) * (c2 * st[3] - (T)2.5));
  if constexpr (NV == 1) {
    g[0] = g0t;
  } else {
    const T eT = dexp(-c2 * st[24]);
    const T g0r = st[25] * eT * ((T)1 + (st[26] * cx + st[27] * cy + st[28] * cz) * (c2 * st[24] - (T)2.5));
    const T g1t = st[29] * g0t + (st[31] * cx + st[32] * cy + st[33] * cz) * et;
    const T g1r = st[30] * g0r + (st[34] * cx + st[35] * cy + st[36] * cz) * eT;
    g[0] = st[37] * g0t + st[38] * g0r;
    g[1] = st[37] * g1t + st[38] * g1r;
  }
}

// state values the kinetic kernels read: Rykov 40; Shakhov 16 (24 with relative storage for
// the loaders of stored f)
template <typename S, int NV>
__host__ __device__ constexpr int stage_state_len() { return NV == 2 ? NST_RYKOV : state_len<S>(); }

// Comparisons on the integer pipe for FP64.  On this GPU an FP64 comparison, min or max holds a
// sub-partition's FP64 pipe as long as an FMA; the bit patterns of IEEE doubles order like their
// values once the magnitude bits of negative values are inverted (sign-magnitude to two's
// complement order), so the comparisons below give the same results on the integer pipe.  FP32
// keeps its native comparisons.
__device__ __forceinline__ long long ordered_key(double x) {
  const long long b = __double_as_longlong(x);
  return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ bool is_greater(double a, double b) { return ordered_key(a) > ordered_key(b); }
__device__ __forceinline__ bool is_greater(float a, float b) { return a > b; }
__device__ __forceinline__ double larger(double a, double b) { return is_greater(a, b) ? a : b; }
__device__ __forceinline__ float larger(float a, float b) { return a > b ? a : b; }
__device__ __forceinline__ double smaller(double a, double b) { return is_greater(a, b) ? b : a; }
__device__ __forceinline__ float smaller(float a, float b) { return a < b ? a : b; }
// a > 0
__device__ __forceinline__ bool is_positive(double a) { return __double_as_longlong(a) > 0; }
__device__ __forceinline__ bool is_positive(float a) { return a > 0.f; }
// a < b for a, b >= 0 (non-negative doubles order like their bit patterns)
__device__ __forceinline__ bool nonneg_lt(double a, double b) { return __double_as_longlong(a) < __double_as_longlong(b); }
__device__ __forceinline__ bool nonneg_lt(float a, float b) { return a < b; }

// Running maximum of non-negative values: of differences (negative ones do not count), of negated
// differences, of magnitudes.  FP64 keeps the bit pattern and compares, negates and clears signs as
// integers: any FP64 instruction, a negation or an absolute value too, costs as much as an FMA.
template <typename T>
struct Largest {
  T v = (T)0;
  __device__ __forceinline__ void raise(T d) { v = fmaxf(v, d); }
  __device__ __forceinline__ void raise_neg(T d) { v = fmaxf(v, -d); }
  __device__ __forceinline__ void raise_abs(T d) { v = fmaxf(v, fabsf(d)); }
  __device__ __forceinline__ T value() const { return v; }
  static __device__ __forceinline__ T least(const Largest &a, const Largest &b) { return fminf(a.v, b.v); }
};
template <>
struct Largest<double> {
  long long v = 0;
  __device__ __forceinline__ void at_least(long long b) { v = b > v ? b : v; }  // (a negative double is a negative integer)
  __device__ __forceinline__ void raise(double d) { at_least(__double_as_longlong(d)); }
  __device__ __forceinline__ void raise_neg(double d) { at_least(__double_as_longlong(d) ^ (long long)0x8000000000000000ULL); }
  __device__ __forceinline__ void raise_abs(double d) { at_least(__double_as_longlong(d) & 0x7fffffffffffffffLL); }
  __device__ __forceinline__ double value() const { return __longlong_as_double(v); }
  static __device__ __forceinline__ double least(const Largest &a, const Largest &b) {
    return __longlong_as_double(a.v < b.v ? a.v : b.v);
  }
};

// Venkatakrishnan limiter of one rectilinear cell: min over its faces (and 1) of
//   (Dm^2 + 2 D2 Dm + e^2) / (Dm^2 + D2 Dm + 2 D2^2 + e^2).
// On each axis |D2| = |g r| is the same on both faces (the centre is the cell's midpoint); one
// meets the bound dp = fmax - fi, the other dn = fi - fmin.  With y = Dm / D2 the function rises in
// y where it is below 1 (y < 2), and at fixed Dm it falls in D2 there (its derivative's sign is that
// of -(Dm^2 + e^2)(4 D2 - Dm) - 4 D2^2 Dm), so the minimum over all faces is the one value at Dm =
// min(dp, dn) and the largest |D2|: with s = Dm + 2 D2, (Dm s + e^2) / (D2 s + Dm^2 + e^2), or 1
// where that is not below 1.  bn / bd is the result.
template <typename T>
__device__ __forceinline__ void venkat_parts(const Largest<T> &dp, const Largest<T> &dn, const Largest<T> &largest_d2, T eps2,
                                             T &bn, T &bd) {
  const T dm = Largest<T>::least(dp, dn), d2 = largest_d2.value();
  const T s = dm + (T)2 * d2;
  bn = dm * s + eps2;
  bd = d2 * s + (dm * dm + eps2);
  if (!nonneg_lt(bn, bd)) bn = bd = (T)1;
}
template <typename T>
__device__ __forceinline__ T venkat_phi(const Largest<T> &dp, const Largest<T> &dn, const Largest<T> &d2, T eps2) {
  T bn, bd;
  venkat_parts<T>(dp, dn, d2, eps2, bn, bd);
  return ddiv(bn, bd);
}

// Per-cell state and colour-entry addresses from 32-bit offsets: a 64-bit multiply by a
// non-power-of-two stride would run at the FP64 rate on this GPU (cells * NST < 2^32 is checked
// at creation).
template <typename T>
__device__ __forceinline__ const T *state_of(const T *st, int cell) {
  return st + (unsigned)cell * (unsigned)NST;
}
__device__ __forceinline__ const EntryInfo &entry_of(const EntryInfo *e, int i) {
  return *reinterpret_cast<const EntryInfo *>(reinterpret_cast<const char *>(e) + (unsigned)i * (unsigned)sizeof(EntryInfo));
}

template <int N = 16>
__device__ __forceinline__ void load_state(const float *__restrict__ src, float *st) {
  const float4 *p = reinterpret_cast<const float4 *>(src);
#pragma unroll
  for (int q = 0; q < N / 4; ++q) {
    const float4 v = __ldg(p + q);
    st[4 * q] = v.x;
    st[4 * q + 1] = v.y;
    st[4 * q + 2] = v.z;
    st[4 * q + 3] = v.w;
  }
}
template <int N = 16>
__device__ __forceinline__ void load_state(const double *__restrict__ src, double *st) {
  const double2 *p = reinterpret_cast<const double2 *>(src);
#pragma unroll
  for (int q = 0; q < N / 2; ++q) {
    const double2 v = __ldg(p + q);
    st[2 * q] = v.x;
    st[2 * q + 1] = v.y;
  }
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

}  // namespace gsis
