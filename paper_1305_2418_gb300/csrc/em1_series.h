// em1_series.h -- e^x - 1 for small x by its Taylor series through x^7/7!, in the type of
// the argument.  At the ends of |x| <= kEm1Small the omitted terms are 1.9e-8 of the
// result; in FP32 the evaluation adds its roundings (below 1.5 ulp in all).  The same
// code compiles as host C++ for testing.
#pragma once
#include <cmath>

#ifdef __CUDACC__
#define EM1_HD __host__ __device__ __forceinline__
#else
#define EM1_HD static inline
#endif

constexpr float kEm1Small = 0.35f;

template <class T>
EM1_HD T em1_series(T x) {
  T q = fma(x, T(1) / T(5040), T(1) / T(720));
  q = fma(x, q, T(1) / T(120));
  q = fma(x, q, T(1) / T(24));
  q = fma(x, q, T(1) / T(6));
  q = fma(x, q, T(0.5));
  return x * fma(x, q, T(1));
}
