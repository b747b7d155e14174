// Values that CTAs of one launch hand to each other (the wavefront block solves
// and the link chain's solves): publication, and bounded waits for it.
#pragma once

#include "ahlp_internal.h"

namespace ahlp {

// Solved entries are their own ready flags: the publication buffers are filled
// with a bit pattern (all ones, a NaN no arithmetic produces) by the first
// kernel of a solve, a writer stores an entry with a relaxed store, a reader
// polls until the pattern is gone.  So a link of the wavefront costs one store
// and one load through L2, where a flag beside the data cost a fence, the flag's
// store and load and then the data's load.
template <typename T>
struct PubBits;
template <>
struct PubBits<float> {
  using U = unsigned;
  static constexpr U none = 0xffffffffu;
  static __device__ __forceinline__ U ld(const float *p) {
    U v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
  }
  static __device__ __forceinline__ void st(float *p, float x) {
    const U v = __float_as_uint(x) == none ? 0x7fffffffu : __float_as_uint(x);
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
  }
  static __device__ __forceinline__ float val(U v) { return __uint_as_float(v); }
};
template <>
struct PubBits<double> {
  using U = unsigned long long;
  static constexpr U none = 0xffffffffffffffffull;
  static __device__ __forceinline__ U ld(const double *p) {
    U v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
  }
  static __device__ __forceinline__ void st(double *p, double x) {
    const U b = (U)__double_as_longlong(x);
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p),
                 "l"(b == none ? 0x7fffffffffffffffull : b)
                 : "memory");
  }
  static __device__ __forceinline__ double val(U v) { return __longlong_as_double((long long)v); }
};

__device__ __forceinline__ int load_relaxed(const int *f) {
  int v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(f) : "memory");
  return v;
}

// Whole-warp bounded wait until no lane's `bits` is the unpublished pattern;
// lanes with `in` reload theirs from p.  Gives up at once when another CTA has
// already timed out, so a failure does not cascade into more waits.
template <typename T>
__device__ __forceinline__ void wait_published(typename PubBits<T>::U &bits, const T *p, bool in,
                                               int *err) {
  using P = PubBits<T>;
  if (!__any_sync(0xffffffffu, in && bits == P::none)) return;
  const unsigned long long t0 = global_ns();
  for (int it = 0;; ++it) {
    if (in && bits == P::none) bits = P::ld(p);
    if (!__any_sync(0xffffffffu, in && bits == P::none)) return;
    if (it >= 8) __nanosleep(64);
    if ((it & 31) == 31) {   // lane 0's clock decides for the warp
      bool out = load_relaxed(err) != 0;
      if (!out && global_ns() - t0 > kWaitLimitNs) {
        atomicExch(err, 1);
        out = true;
      }
      if (__shfl_sync(0xffffffffu, out ? 1 : 0, 0)) return;
    }
  }
}

}  // namespace ahlp
