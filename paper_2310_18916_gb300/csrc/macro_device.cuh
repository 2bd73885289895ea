// macro_device.cuh -- device helpers shared by the two synthetic solves (macro.cu, macro_general.cu).
#pragma once
#include <cuda_runtime.h>

#include "fp64_device.cuh"
#include "gsis_internal.h"

namespace gsis {
namespace {
constexpr long long kSpinLimit = 1LL << 31;  // ~1 s of clock64 cycles at 2 GHz

constexpr int kBarGroups = 8, kBarStride = 32;  // arrival counters, 128 bytes apart
static_assert(kBarGroups * kBarStride <= MACRO_BAR_WORDS, "barrier words");

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void red_release_add(unsigned *p, unsigned x) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(x) : "memory");
}

// block barrier of the first nthreads threads (a multiple of 32)
__device__ __forceinline__ void block_part_sync(int nthreads) { asm volatile("bar.sync 1, %0;" ::"r"(nthreads) : "memory"); }

// Grid barrier on kBarGroups monotonic arrival counters, each in its own 128-byte line and zero
// at launch.  Block b adds 1 to counter b % kBarGroups with release semantics (publishing the
// block's writes); thread g < kBarGroups of every block waits, with acquire loads, until counter
// g has reached the barrier's epoch (1, 2, ...) times its group size.  Spreading the arrivals
// keeps same-address atomics from serialising on one line.  The spin is bounded: on time-out
// it raises the error flag.  Returns false when a block has flagged an error; the flag is read while
// the counters are polled (after them it cost another L2 round trip, 460 to 830 of about 5000
// cycles), so an error raised just before another block's arrival may show at the next barrier
// only: a block that left is then missed there, and the polls end on the flag.
__device__ __forceinline__ bool barrier_wait(unsigned *bar, unsigned epoch, int *err, long long limit) {
  bool bad = false;
  if (threadIdx.x == 0) red_release_add(bar + kBarStride * (blockIdx.x % kBarGroups), 1u);
  if (threadIdx.x < kBarGroups) {
    const unsigned g = threadIdx.x, gsize = (gridDim.x - g + kBarGroups - 1) / kBarGroups;
    const unsigned target = epoch * gsize;
    const long long t0 = clock64();
    for (unsigned i = 0; ld_acquire(bar + kBarStride * g) < target; ++i) {
      if ((i & 15u) == 15u && (clock64() - t0 > limit || *(volatile int *)err != 0)) {
        atomicCAS(err, 0, GSIS_ERR_TIMEOUT);
        bad = true;
        break;
      }
      __nanosleep(32);
    }
  } else if (threadIdx.x == 32) {
    bad = *(volatile int *)err != 0;
  }
  return bad;
}

__device__ bool grid_sync(unsigned *bar, unsigned &epoch, int *err, long long limit = kSpinLimit) {
  ++epoch;
  __syncthreads();
  return !__syncthreads_or(barrier_wait(bar, epoch, err, limit));
}

// The barrier of the first nthreads (a multiple of 32) threads of every block, which alone call it; the
// other warps' epoch is advanced by the caller and an error shows at the next full barrier.
__device__ __forceinline__ void grid_sync_part(unsigned *bar, unsigned &epoch, int *err, int nthreads) {
  ++epoch;
  block_part_sync(nthreads);
  barrier_wait(bar, epoch, err, kSpinLimit);
  block_part_sync(nthreads);
}

// Comparisons on the integer pipe (an FP64 comparison, min or max costs as much as an FMA on this
// GPU).  Where the operands are known to be non-negative, the order of their bit patterns as
// integers is their numeric order (no NaN reaches them on a physical state).
// x > 0 exactly as the FP64 comparison: +0 < bits <= +inf (negative values, -0 and NaN fail)
__device__ __forceinline__ bool gt0(double x) {
  return (unsigned long long)(dbits(x) - 1) < 0x7ff0000000000000ULL;
}
// x < y and max(x, y) for x, y >= 0
__device__ __forceinline__ bool lt_nn(double x, double y) { return dbits(x) < dbits(y); }
__device__ __forceinline__ double max_nn(double x, double y) { return dbits(x) < dbits(y) ? y : x; }

__device__ __forceinline__ double sound(double Tt) { return root(Tt * (5.0 / 6.0)); }

// A value with the number of the pass that wrote it, one 16-byte access (a single copy)
__device__ __forceinline__ void st_tagged(double *p, double v, unsigned long long tag) {
  asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p),
               "l"(__double_as_longlong(v)), "l"(tag)
               : "memory");
}
// loads both where `want` is not 0, else leaves them; does not branch, so that several are in flight
__device__ __forceinline__ void ld_tagged_if(unsigned want, const double *p, double *v, unsigned long long *tag) {
  long long x = __double_as_longlong(*v);
  asm volatile(
      "{\n\t.reg .b128 t;\n\t.reg .pred q;\n\tsetp.ne.u32 q, %3, 0;\n\tmov.b128 t, {%0, %1};\n\t"
      "@q ld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
      : "+l"(x), "+l"(*tag)
      : "l"(p), "r"(want)
      : "memory");
  *v = __longlong_as_double(x);
}

// Polls for N published terms (this lane's bits of `need`), each until it carries its tag (src and
// tag of term f), all that are still missing in one round trip (a branch per term takes them one
// after the other).  The whole warp takes part; bounded: on time-out, or once any block has flagged
// an error, it raises the flag and returns (every block then leaves at its next grid barrier).
template <int N, typename Src, typename Tag>
__device__ __forceinline__ void await_terms(unsigned need, Src src, Tag tag_of, double *v, int *err) {
  unsigned long long tag[N];
#pragma unroll
  for (int f = 0; f < N; ++f) {
    v[f] = 0.0;
    tag[f] = ~0ULL;
  }
  unsigned miss = need;
  const long long t0 = clock64();
  for (unsigned it = 0;; ++it) {
#pragma unroll
    for (int f = 0; f < N; ++f) ld_tagged_if(miss >> f & 1, src(f), v + f, tag + f);
#pragma unroll
    for (int f = 0; f < N; ++f)
      if (tag[f] == tag_of(f)) miss &= ~(1u << f);
    if (!__any_sync(0xffffffffu, miss != 0)) return;
    if ((it & 31u) == 31u) {
      const bool quit = clock64() - t0 > kSpinLimit || *(volatile int *)err != 0;
      if (__any_sync(0xffffffffu, quit)) {
        if ((threadIdx.x & 31) == 0) atomicCAS(err, 0, GSIS_ERR_TIMEOUT);
        return;
      }
    }
  }
}
}  // namespace
}  // namespace gsis
