// Sums of FP32 products to about twice FP32's precision on the FP32 pipe (FP64 runs at 1/64 of its rate):
// error-free transformations after Knuth (two-sum) and Dekker (product error, here by fma).
#pragma once

namespace ks {

struct SumPair {
  float s = 0.f, c = 0.f;                                            // s + c, |c| of the order of s's rounding
  // x + e, |e| of the order of x's rounding
  __device__ __forceinline__ void add(float x, float e) {
    const float t = s + x, bp = t - s;
    c += ((s - (t - bp)) + (x - bp)) + e;
    s = t;
  }
  __device__ __forceinline__ void add_product(float a, float b) {
    const float p = a * b;
    add(p, fmaf(a, b, -p));
  }
  __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};

}  // namespace ks
