// Sums of many T values in at least FP64 precision (sm_103a).
//
// FP64 path: plain.  FP32 path: the chip has 2 FP64 lanes per SM and cycle, so a conversion and an
// FP64 add cost 16 cycles of an SM each per warp instruction.  Here the sum is three floats, each
// collecting the exact rounding errors of the one before (Knuth's two-sum): 13 FP32 operations,
// 3.3 cycles.  hi and mid lose nothing; lo rounds at 2^-24 of itself, below 2^-65 of the sum of
// the magnitudes for up to 128 terms, where an FP64 sum rounds at 2^-53 with every term.  (Two
// floats round at 2^-48 and below with every term: less than FP64.)
#pragma once
#include "common.cuh"

namespace ll {

template <typename T> struct DSum;
template <> struct DSum<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double v) { s += v; }
  __device__ __forceinline__ double value() const { return s; }
};
template <> struct DSum<float> {
  float hi = 0.f, mid = 0.f, lo = 0.f;
  // a += b; returns the exact rounding error
  static __device__ __forceinline__ float two_sum(float& a, float b) {
    const float s = __fadd_rn(a, b), t = __fadd_rn(s, -a);
    const float e = __fadd_rn(__fadd_rn(a, -__fadd_rn(s, -t)), __fadd_rn(b, -t));
    a = s;
    return e;
  }
  __device__ __forceinline__ void add(float v) { lo = __fadd_rn(lo, two_sum(mid, two_sum(hi, v))); }
  __device__ __forceinline__ double value() const {   // not finite: hi is what a plain sum is
    return fabsf(hi) <= 3.402823466e38f ? (double)hi + ((double)mid + (double)lo) : (double)hi;
  }
};

}  // namespace ll
