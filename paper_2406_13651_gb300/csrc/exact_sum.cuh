// exact_sum.cuh -- four FP32 values into an FP64 sum, with FP64's rounding only.
//
// Of FP64 operations an SM does two a clock, so four values are first added in FP32 without error
// (two-sum: Knuth, The Art of Computer Programming 2, 4.2.2): head + middle + rest is their exact sum, the
// head and the middle take one FP64 addition each, and the rest is nearly always zero.
#pragma once
#include <math.h>

#if !defined(__CUDACC__)
#define __host__
#define __device__
#endif

namespace clamp {

// a + b rounded, with e = a + b - (a + b rounded) exactly (finite results).
__host__ __device__ inline float two_sum(float a, float b, float& e) {
  const float t = a + b, bp = t - a;
  e = (a - (t - bp)) + (b - bp);
  return t;
}

__host__ __device__ inline void add_four(double& acc, float a, float b, float c, float d) {
  float e0, e1, e2, f1, f2;
  const float s0 = two_sum(a, b, e0), s1 = two_sum(c, d, e1), head = two_sum(s0, s1, e2);
  if (isfinite(head)) {
    const float m = two_sum(e0, e1, f1), middle = two_sum(e2, m, f2);
    acc += (double)head;
    acc += (double)middle;
    if (f1 != -f2) acc += (double)f1 + (double)f2;
  } else {   // a value that is not finite, or a sum beyond FP32
    acc += ((double)a + b) + ((double)c + d);
  }
}

}  // namespace clamp
