// A quotient from the divisor's reciprocal, with the bits of the division.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>
#include <cstring>

namespace sharpy {

__host__ __device__ __forceinline__ uint64_t double_bits(double x) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t b;
  std::memcpy(&b, &x, 8);
  return b;
#endif
}
__host__ __device__ __forceinline__ double bits_double(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double x;
  std::memcpy(&x, &b, 8);
  return x;
#endif
}

// t / c from c's correctly rounded reciprocal r (Markstein, IBM J. Res. Dev.
// 34, 1990): with q within an ulp of t / c, q + (t - q c) r in fused operations
// is the correctly rounded quotient, the bits of t / c. The first step brings
// q = t r there, the second rounds: 5 operations that share one reciprocal
// over a column. A zero loses its sign on the way: it is t r's. Outside the
// exponent range where that holds (of c too: 0 / inf is 0, 0 times anything with
// inf is not) it divides.
__host__ __device__ __forceinline__ double quotient(double t, double c, double r) {
  const uint64_t bt = double_bits(t);
  const int ht = (int)(bt >> 32) & 0x7fffffff, hr = (int)(double_bits(r) >> 32) & 0x7fffffff;
  const double q = t * r;
  const uint64_t bq = double_bits(q);
  const int hq = (int)(bq >> 32) & 0x7fffffff;
  constexpr int lo = 200 << 20, hi = 1846 << 20;
  if (hr > lo && hr < hi && ((ht > lo && ht < hi && hq > lo && hq < hi) || (ht | (int)(uint32_t)bt) == 0)) {
    const double q1 = fma(fma(-q, c, t), r, q);
    const double q2 = fma(fma(-q1, c, t), r, q1);
    return bits_double(double_bits(q2) | (bq & 0x8000000000000000ULL));
  }
  return t / c;
}

}  // namespace sharpy
