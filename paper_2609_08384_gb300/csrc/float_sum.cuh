// Sum of a few floats in two: the rounding error of every addition (Knuth's two-sum)
// is added up in lo, so hi + lo carries n terms to n^2 2^-50.  For short sums that go on
// into an FP64 accumulator: over 16384 equal terms lo itself rounds, and the sum came
// out 2^-25 off.  FP64 operations are scarce on this GPU (about two lanes per SM and
// cycle): a convert and an add per pair of points made the FP64 pipe the bound of the
// power trace: 149 us on the 403 MB of 3 x 512x512x64, with two of each per eight pairs
// 101 (with one two-float sum per thread 96).
// A sum beyond FP32's range comes out infinite or undefined; callers then add the
// terms one by one in FP64.
#pragma once

#include <cuda_runtime.h>

namespace brahms {

struct FloatSum {
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float t = __fadd_rn(hi, x);
    const float z = __fsub_rn(t, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(t, z)), __fsub_rn(x, z)));
    hi = t;
  }
  __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

}  // namespace brahms
