// stencil_int.cuh -- the linear stencils of Eqs. 6-7 on binary64 values by
// integer arithmetic.
//
// GB300 retires 1.7 binary64 operations a clock and SM against 64 32-bit
// integer ones, so a binary64 instruction costs a warp as much as some 38
// integer ones.  The weights of the stencils are small integers up to a common
// factor (8, 1 and 16, 1, 30 times 1/(12 h) and 1/(12 h^2)), so their sums
// need no multiplications: the values are aligned to the largest exponent among
// them as 64-bit integers with four guard bits, summed exactly, and the sum is
// rounded once, to nearest.  Values within a factor of 16 of the largest lose
// nothing; the others are cut at 2^-56 of its power of two.  A result is thus within
// half a unit of its own last place and as many of those cuts as the weights add
// up to: 18 (first derivative), 34 or 64 (second, without and with the centre), 36
// (first of eight values).  That is an error in terms of the largest value, as
// those of binary64 operations are in terms of the largest partial sum: on four
// values uniform in +-1 the first derivative's is 3.8e-16 of the largest value rms and
// 2.0e-15 at most, against 5.0e-16 and 3.4e-15 of binary64 operations, on neighbours of a
// smooth function as large or half as large.  But where the large values cancel
// exactly and far smaller ones are left, binary64 keeps those and this does not: (1, 0, 1e-17, 1)
// gives 0 for 8e-17.  Zeros are exact and odd symmetry is kept (f -> -f).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

namespace sbli {

namespace fixed {

__host__ __device__ __forceinline__ uint32_t high(double x) {
#ifdef __CUDA_ARCH__
  return (uint32_t)__double2hiint(x);
#else
  uint64_t b;
  memcpy(&b, &x, 8);
  return (uint32_t)(b >> 32);
#endif
}
__host__ __device__ __forceinline__ uint32_t low(double x) {
#ifdef __CUDA_ARCH__
  return (uint32_t)__double2loint(x);
#else
  uint64_t b;
  memcpy(&b, &x, 8);
  return (uint32_t)b;
#endif
}
__host__ __device__ __forceinline__ double from_bits(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double x;
  memcpy(&x, &b, 8);
  return x;
#endif
}
// shifts by 64 and more give 0
__host__ __device__ __forceinline__ uint64_t shr(uint64_t v, uint32_t s) {
#ifdef __CUDA_ARCH__
  uint64_t r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
  return r;
#else
  return s > 63 ? 0 : v >> s;
#endif
}
__host__ __device__ __forceinline__ uint32_t leading_zeros(uint64_t v) {  // v != 0
#ifdef __CUDA_ARCH__
  return (uint32_t)__clzll((long long)v);
#else
  return (uint32_t)__builtin_clzll(v);
#endif
}

constexpr uint32_t EXPONENT = 0x7FF00000u;

// The exponent field (in place) that values are aligned to: the largest
// among them, but at least 66, so that zeros and subnormals (which lack the
// implied leading bit) are shifted out; values below 2^-957 are thereby cut at
// 2^-1013.
template <typename... V>
__host__ __device__ __forceinline__ uint32_t top_exponent(double x, V... rest) {
  const uint32_t e = high(x) & EXPONENT;
  uint32_t r = 66u << 20;
  if constexpr (sizeof...(rest) > 0) r = top_exponent(rest...);
  return e > r ? e : r;
}
// Whether values with this largest exponent can be aligned: neither infinite,
// NaN nor so large that a sum may overflow.
__host__ __device__ __forceinline__ bool alignable(uint32_t top) { return top < (2032u << 20); }
// x in units of 2^-56 of the largest exponent
__host__ __device__ __forceinline__ int64_t aligned(double x, uint32_t top) {
  const uint32_t h = high(x);
  const uint32_t s = (top - (h & EXPONENT)) >> 20;
  uint64_t m = ((uint64_t)((h & 0xFFFFFu) | 0x100000u) << 32) | low(x);
  m = shr(m << 4, s);
  const int64_t sign = (int64_t)((int32_t)h >> 31);
  return (int64_t)(m ^ (uint64_t)sign) - sign;
}
// v units of 2^-56 of the exponent `top` as binary64, rounded to nearest (ties
// away from zero)
__host__ __device__ __forceinline__ double rounded(int64_t v, uint32_t top) {
  const uint64_t sign = (uint64_t)v & 0x8000000000000000ull;
  uint64_t m = v < 0 ? 0 - (uint64_t)v : (uint64_t)v;
  const uint32_t n = leading_zeros(m | 1u);
  m <<= n;
  const uint32_t e = top + (6u << 20) - (n << 20);  // one less: the leading bit of m adds one
  const uint64_t b = ((uint64_t)e << 32) + (m >> 11) + ((m >> 10) & 1u);
  return from_bits(v == 0 ? 0 : b | sign);
}

}  // namespace fixed

// The stencils on values at offsets -2, -1, +1, +2.  FIXED: in integers, given the
// values' top exponent (alignable); otherwise in binary64.
// 8 (p1 - m1) - (p2 - m2): times 1/(12 h) the first derivative of Eq. 6
template <bool FIXED>
__host__ __device__ __forceinline__ double first_sum(double m2, double m1, double p1, double p2, uint32_t top) {
  if constexpr (!FIXED) return 8.0 * (p1 - m1) - (p2 - m2);
  const int64_t a = fixed::aligned(p1, top) - fixed::aligned(m1, top);
  const int64_t b = fixed::aligned(p2, top) - fixed::aligned(m2, top);
  return fixed::rounded((int64_t)((uint64_t)a << 3) - b, top);
}
// the same of the sums x + y, top that of all eight values
template <bool FIXED>
__host__ __device__ __forceinline__ double first_sum(const double (&x)[4], const double (&y)[4], uint32_t top) {
  if constexpr (!FIXED) return 8.0 * ((x[2] + y[2]) - (x[1] + y[1])) - ((x[3] + y[3]) - (x[0] + y[0]));
  int64_t v[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) v[k] = fixed::aligned(x[k], top) + fixed::aligned(y[k], top);
  return fixed::rounded((int64_t)((uint64_t)(v[2] - v[1]) << 3) - (v[3] - v[0]), top);
}
// (p2 + m2) - 16 (p1 + m1): times -1/(12 h^2) the second derivative of Eq. 7
// without its centre term
template <bool FIXED>
__host__ __device__ __forceinline__ double second_sum(double m2, double m1, double p1, double p2, uint32_t top) {
  if constexpr (!FIXED) return (p2 + m2) - 16.0 * (p1 + m1);
  const int64_t a = fixed::aligned(p1, top) + fixed::aligned(m1, top);
  const int64_t b = fixed::aligned(p2, top) + fixed::aligned(m2, top);
  return fixed::rounded(b - (int64_t)((uint64_t)a << 4), top);
}
// both, the values aligned once
template <bool FIXED>
__host__ __device__ __forceinline__ void both_sums(double m2, double m1, double p1, double p2, uint32_t top,
                                                   double& first, double& second) {
  if constexpr (!FIXED) {
    first = first_sum<false>(m2, m1, p1, p2, top);
    second = second_sum<false>(m2, m1, p1, p2, top);
    return;
  }
  const int64_t a = fixed::aligned(p1, top), b = fixed::aligned(m1, top);
  const int64_t x = fixed::aligned(p2, top), y = fixed::aligned(m2, top);
  first = fixed::rounded((int64_t)((uint64_t)(a - b) << 3) - (x - y), top);
  second = fixed::rounded((x + y) - (int64_t)((uint64_t)(a + b) << 4), top);
}

__host__ __device__ __forceinline__ double stencil_first(double m2, double m1, double p1, double p2) {
  const uint32_t top = fixed::top_exponent(m2, m1, p1, p2);
  return fixed::alignable(top) ? first_sum<true>(m2, m1, p1, p2, top) : first_sum<false>(m2, m1, p1, p2, top);
}
// 16 (p1 + m1) - (p2 + m2) - 30 c: times 1/(12 h^2) the second derivative of Eq. 7
__host__ __device__ __forceinline__ double stencil_second(double m2, double m1, double c, double p1, double p2) {
  const uint32_t top = fixed::top_exponent(m2, m1, c, p1, p2);
  if (!fixed::alignable(top)) return (16.0 * (p1 + m1) - (p2 + m2)) - 30.0 * c;
  const int64_t a = fixed::aligned(p1, top) + fixed::aligned(m1, top);
  const int64_t b = fixed::aligned(p2, top) + fixed::aligned(m2, top);
  const int64_t v = fixed::aligned(c, top);
  return fixed::rounded((int64_t)((uint64_t)a << 4) - b - (int64_t)(((uint64_t)v << 5) - ((uint64_t)v << 1)), top);
}
// both, the values aligned once where the centre does not raise the exponent that
// the first derivative's values are aligned to (else each by itself)
__host__ __device__ __forceinline__ void stencil_both(double m2, double m1, double c, double p1, double p2,
                                                      double& first, double& second) {
  const uint32_t top = fixed::top_exponent(m2, m1, p1, p2);
  if (!fixed::alignable(top) || (fixed::high(c) & fixed::EXPONENT) > top) {
    first = stencil_first(m2, m1, p1, p2);
    second = stencil_second(m2, m1, c, p1, p2);
    return;
  }
  const int64_t ap = fixed::aligned(p1, top), am = fixed::aligned(m1, top), v = fixed::aligned(c, top);
  const int64_t bp = fixed::aligned(p2, top), bm = fixed::aligned(m2, top);
  first = fixed::rounded((int64_t)((uint64_t)(ap - am) << 3) - (bp - bm), top);
  second = fixed::rounded(
      (int64_t)((uint64_t)(ap + am) << 4) - (bp + bm) - (int64_t)(((uint64_t)v << 5) - ((uint64_t)v << 1)), top);
}

}  // namespace sbli
