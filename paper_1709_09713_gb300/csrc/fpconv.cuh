// fpconv.cuh -- binary32 <-> binary64 conversions without the FP64 pipe.
//
// GB300 executes F2F.F64.F32 / F2F.F32.F64 on its (narrow) FP64 pipe at the
// DFMA rate, about 2 per clock per SM.  The binary32-storage stage converts
// every stage value and accumulator increment, and the double-float one splits
// every stage field, so these re-pack the IEEE bit patterns with integer operations
// instead; each states how it rounds and what becomes of subnormals, infinities and
// NaNs.
#pragma once

#include <cuda_runtime.h>

namespace sbli {

// Branch-free forms used in the stage kernels.  widen_f32_fast equals the
// hardware conversion except that binary32 subnormal inputs become signed
// zero; narrow_f64_fast equals __double2float_rn except that inputs of
// magnitude below 2^-126 become signed zero and NaNs become one quiet NaN.
__device__ __forceinline__ double widen_f32_fast(float x) {
  const unsigned u = __float_as_uint(x);
  const unsigned e = u & 0x7F800000u;
  const unsigned sign = u & 0x80000000u;
  unsigned hi = (((u & 0x7FFFFFFFu) >> 3) + 0x38000000u) | sign;
  unsigned lo = u << 29;
  hi = (e == 0u) ? sign : hi;
  lo = (e == 0u) ? 0u : lo;
  hi = (e == 0x7F800000u) ? (hi | 0x7FF00000u) : hi;
  return __hiloint2double((int)hi, (int)lo);
}

__device__ __forceinline__ float narrow_f64_fast(double d) {
  const unsigned hi = (unsigned)__double2hiint(d);
  const unsigned lo = (unsigned)__double2loint(d);
  const unsigned sign = hi & 0x80000000u;
  const unsigned eb = (hi >> 20) & 0x7FFu;
  const unsigned mant = ((hi & 0xFFFFFu) << 3) | (lo >> 29);
  unsigned bits = sign | ((eb - 896u) << 23) | mant;
  const unsigned rest = lo & 0x1FFFFFFFu;
  bits += (rest > 0x10000000u || (rest == 0x10000000u && (bits & 1u))) ? 1u : 0u;
  bits = (eb < 897u) ? sign : bits;                      // zero / below the binary32 normal range
  bits = (eb > 1150u) ? (sign | 0x7F800000u) : bits;     // overflow and infinity
  bits = (eb == 0x7FFu && (((hi & 0xFFFFFu) | lo) != 0u)) ? 0x7FFFFFFFu : bits;  // NaN
  return __uint_as_float(bits);
}

// The narrowing of the binary32 stage values and of the binary32 copy of
// the state (binary32 stages with a binary64 accumulator): round to nearest,
// ties away from zero (the same error bound as ties-to-even, half a unit in
// the last place).  One funnel shift brings the 23 kept mantissa bits and the
// low 9 exponent bits together; adding 0x40000000 rebases the exponent
// (e - 896, taken modulo 2^9, lands in bits 30..23 with bit 31 clear for
// every binary32-normal result); the first dropped bit is the rounding
// increment, whose carry moves into the exponent when the mantissa
// overflows.  Results below the binary32 normal range are signed zero;
// magnitudes of 2^128 and above, infinities and NaNs give signed infinity (a
// NaN stays NaN in the binary64 accumulator and state).
__device__ __forceinline__ float narrow_f64_rna(double d) {
  const unsigned hi = (unsigned)__double2hiint(d);
  const unsigned lo = (unsigned)__double2loint(d);
  const unsigned t = __funnelshift_l(lo, hi, 3) + 0x40000000u + ((lo >> 28) & 1u);
  const unsigned sign = hi & 0x80000000u;
  const unsigned eb = (hi >> 20) & 0x7FFu;
  unsigned bits = t | sign;
  bits = (eb < 897u) ? sign : bits;
  bits = (eb > 1150u) ? (sign | 0x7F800000u) : bits;
  return __uint_as_float(bits);
}

// 1/x in binary64: the hardware approximation y (rcp.approx.ftz.f64, 20 bits)
// refined in one step of third order, y (1 + e + e^2) with e = 1 - x y, whose relative
// error e^3 is below 2^-59: three fused multiply-adds where two Newton-Raphson
// steps take four (within one unit in the last place of 1/x;
// tests/test_gpu_recip.py compares it with CUDA's correctly rounded reciprocal)
__device__ __forceinline__ double rcp_newton_f64(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// x / y, given 1/y: the product corrected by its residual (Markstein), so that it
// rounds as the division does
__device__ __forceinline__ double corrected_quotient(double x, double y, double yinv) {
  const double q = x * yinv;
  return fma(fma(-q, y, x), yinv, q);
}

// binary64 -> double-float pair, hi = v rounded to nearest (ties away from
// zero), lo = v - hi rounded to nearest, without the FP64 pipe: the low word
// shifted left by 3 holds the 29 mantissa bits that hi drops at the top of a
// signed integer, which is negative just when hi was rounded up -- the exact
// remainder in units of 2^(e - 55); converted (one rounding, to 24 bits) and
// scaled by that power of two with the sign of v, in two exact steps, as 2^(e - 55)
// itself leaves the binary32 range at 2^-71 where lo does not (in one step, 24 bits
// below 2^-71, a double-float solve took 2.30 instead of 2.31 ms at 129x97x66, 16.96
// either way at 256^3).  Zero and results below the binary32 normal range become
// signed zero, lo as well as hi, so a pair holds its value to 48 bits or to 2^-126;
// magnitudes of 2^128 and above and infinities give an infinite hi, NaNs a NaN,
// with lo 0.
// The stage kernels split binary64 stage inputs this way, and the
// double-float path stores its stage fields already split this way.
__device__ __forceinline__ void split_f64(double v, float& hi, float& lo) {
  const unsigned vh = (unsigned)__double2hiint(v), vl = (unsigned)__double2loint(v);
  const unsigned sign = vh & 0x80000000u, eb = (vh >> 20) & 0x7FFu;
  unsigned bits = (__funnelshift_l(vl, vh, 3) + 0x40000000u + ((vl >> 28) & 1u)) | sign;
  unsigned scale = sign | ((eb - 920u) << 23);  // 2^(e - 24), biased: eb - 1023 + 127 - 24
  const float rest = __fmul_rn(__int2float_rn((int)(vl << 3)), 0x1p-31f);
  bits = eb < 897u ? sign : bits;
  scale = eb < 921u ? sign : scale;  // |lo| <= 2^(e - 24), below the normal range
  if (eb > 1150u) {  // 2^128 and above, infinities, NaNs
    bits = sign | 0x7F800000u | (eb == 0x7FFu && ((vh & 0xFFFFFu) | vl) != 0u ? 0x400000u : 0u);
    scale = 0u;
  }
  hi = __uint_as_float(bits);
  asm("mul.rn.ftz.f32 %0, %1, %2;" : "=f"(lo) : "f"(rest), "f"(__uint_as_float(scale)));
}

}  // namespace sbli
