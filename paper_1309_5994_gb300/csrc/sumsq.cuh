// Sum of squares of FP32 values in two FP32 words (about 46 bits): the FP64 pipe has no room for an addition per
// element, and one FP32 word would lose the low bits of a norm that decides about orthogonality.  Dekker's product
// error by an FMA and Knuth's two-sum (a compiler that contracts hi + x x to one FMA leaves the same total).  Plain C++, so that it compiles without the CUDA headers too.
#pragma once
#include <cmath>

#ifdef __CUDACC__
#define SUMSQ_HD __host__ __device__ __forceinline__
#else
#define SUMSQ_HD inline
#endif

struct SumSq {
  float hi = 0.f, lo = 0.f;
  SUMSQ_HD void add(float x) {
    const float p = x * x, e = fmaf(x, x, -p);
    const float s = hi + p, b = s - hi;
    lo += e + ((hi - (s - b)) + (p - b));
    hi = s;
  }
  SUMSQ_HD double value() const { return (double)hi + (double)lo; }
};
