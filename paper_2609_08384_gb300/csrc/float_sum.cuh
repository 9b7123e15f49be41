// Running sum of floats without loss: the rounding error of every addition
// (Knuth's two-sum) is kept in a second float, so hi + lo carries about 2^-45 of
// the sum through thousands of terms.  FP64 additions are scarce on this GPU
// (about two lanes per SM and cycle): a convert and an add per pair of points made
// the FP64 pipe the bound of the power trace (230 us on 805 MB, 143 this way).
// A sum beyond FP32's range comes out infinite or undefined; callers then add the
// terms again in FP64.  (Moving large sums to FP64 inside add() cost every
// addition its predicated FP64 instructions: 440 us.)
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
