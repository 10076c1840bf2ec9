// Sum of FP32 terms in three FP32 words, for reductions whose FP64 form is bound by the FP64 pipe (a conversion and an
// addition per term, at a small fraction of the FP32 rate).  Each word takes the exact rounding error of the word above it
// (Knuth's two-sum); only the third is rounded.  What is lost is of order 2^-72 of the largest running sum per term, where a
// chain of FP64 additions loses 2^-53; two words alone lose 2^-48.  A sum whose words are not all finite has left FP32's
// range on the way and has to be taken again in FP64.
#pragma once
#include <math.h>

#ifdef __CUDACC__
#define FR3D_HD __host__ __device__ __forceinline__
#else
#define FR3D_HD inline
#endif

namespace fr3d {

struct WideSum {
  float w[3] = {0.f, 0.f, 0.f};
  // a + b rounded; b becomes the rounding error
  static FR3D_HD float two_sum(float a, float& b) {
    const float s = a + b, d = s - a;
    b = (a - (s - d)) + (b - d);
    return s;
  }
  FR3D_HD void add(float x) {
    w[0] = two_sum(w[0], x);
    w[1] = two_sum(w[1], x);
    w[2] += x;
  }
  FR3D_HD bool finite() const { return isfinite(w[0]) && isfinite(w[1]) && isfinite(w[2]); }
  FR3D_HD double value() const { return (double)w[0] + ((double)w[1] + (double)w[2]); }
};

}  // namespace fr3d
