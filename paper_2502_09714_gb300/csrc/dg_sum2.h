// Compensated sums of FP32 terms (the adjoint's scalars): as exact as an FP64 accumulator for the few hundred terms
// that one takes, without the FP64 units.
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define DG_SUM2_FN __host__ __device__ __forceinline__
#else
#define DG_SUM2_FN inline
#endif

namespace dg {

// Knuth's two-sum; the rounding errors are collected in lo.
struct Sum2 {
  float hi, lo;
  DG_SUM2_FN explicit Sum2(float x, float e = 0.f) : hi(x), lo(e) {}
  DG_SUM2_FN Sum2& add(float x) {
    const float t = hi + x, b = t - hi;
    lo += (hi - (t - b)) + (x - b);
    hi = t;
    return *this;
  }
  DG_SUM2_FN Sum2& add(const Sum2& x) {
    add(x.hi);
    lo += x.lo;
    return *this;
  }
  DG_SUM2_FN Sum2& scale(float k) {
    const float p = hi * k;
    lo = fmaf(lo, k, fmaf(hi, k, -p));
    hi = p;
    return *this;
  }
  DG_SUM2_FN float value() const { return hi + lo; }
  DG_SUM2_FN double wide() const { return static_cast<double>(hi) + static_cast<double>(lo); }
};

// Sum of the terms k = q, q + 4, .. < n of n floats st apart: a quarter of them, for one of four threads.
DG_SUM2_FN Sum2 quarter_sum(const float* p, int n, int st, int q) {
  Sum2 s(0.f);
  for (int k = q; k < n; k += 4) s.add(p[k * st]);
  return s;
}

}  // namespace dg

#undef DG_SUM2_FN
