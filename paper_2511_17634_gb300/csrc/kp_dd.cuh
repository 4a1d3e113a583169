// kp_dd.cuh -- double-float ("dd") arithmetic on the FP32 pipe.
//
// A value is the unevaluated sum hi + lo of two floats (about 48 significant
// bits).  GB300 issues about 2 FP64 operations per clock per SM against 128
// FP32 ones, so the solvers' high-precision true residuals run in this form:
// a dd add or multiply costs 7-11 FP32 instructions, several times less issue
// time than one FP64 instruction.
//
// The building blocks are the classical error-free transformations:
//  * TwoSum (Knuth): s = fl(a + b) and the exact error e, a + b = s + e;
//  * Fast-TwoSum (Dekker), for |a| >= |b|: the same in three operations;
//  * TwoProduct with a fused multiply-add: p = fl(a b), e = fma(a, b, -p).
// dd_add is the "sloppy" sum (hi parts by TwoSum, lo parts added, one
// renormalisation): its error is bounded by a few units of 2^-44 times
// |x| + |y|, i.e. relative to the operands, not to the result -- the bound a
// residual b - A x needs, whose accuracy is judged against ||b||.
//
// FP64 <-> dd conversions: dd_from_double splits the FP64 bit pattern with
// integer operations (no FP64 instruction): hi = x truncated to 24
// significant bits, lo = the remaining 29 bits rounded to 24; below 2^-100 both
// are zero, far under any quantity the solvers compare.  |x| >= 2^128, an
// infinity or NaN leaves an infinity or NaN in lo (hi is then meaningless),
// which every sum of the low parts carries on: marking hi as well, by a
// compare and two selects per value, made the mixed-precision solves 3 to 8 %
// slower.  dd_to_double rounds hi + lo to FP64 (exact up to 53 significant
// bits); dd_to_double_any does so for such values too.
#pragma once

#include <cuda_runtime.h>

namespace kp {

struct dd {
  float hi, lo;
};

__device__ __forceinline__ dd dd_two_sum(float a, float b) {
  const float s = a + b;
  const float bb = s - a;
  const float e = (a - (s - bb)) + (b - bb);
  return {s, e};
}

__device__ __forceinline__ dd dd_fast_two_sum(float a, float b) {
  const float s = a + b;
  return {s, b - (s - a)};
}

__device__ __forceinline__ dd dd_add(dd x, dd y) {
  dd s = dd_two_sum(x.hi, y.hi);
  s.lo += x.lo + y.lo;
  return dd_fast_two_sum(s.hi, s.lo);
}

__device__ __forceinline__ dd dd_sub(dd x, dd y) { return dd_add(x, dd{-y.hi, -y.lo}); }

__device__ __forceinline__ dd dd_add_f(dd x, float y) {
  dd s = dd_two_sum(x.hi, y);
  s.lo += x.lo;
  return dd_fast_two_sum(s.hi, s.lo);
}

__device__ __forceinline__ dd dd_mul(dd x, dd y) {
  const float p = __fmul_rn(x.hi, y.hi);   // (never contracted with the sum below)
  float e = fmaf(x.hi, y.hi, -p);
  e = fmaf(x.hi, y.lo, e);
  e = fmaf(x.lo, y.hi, e);
  return dd_fast_two_sum(p, e);
}

__device__ __forceinline__ dd dd_from_double(double x) {
  const unsigned int uh = (unsigned int)__double2hiint(x), ul = (unsigned int)__double2loint(x);
  const unsigned int sign = uh & 0x80000000u, mag = uh ^ sign;
  const int e = (int)(mag >> 20);                    // biased FP64 exponent
  // top 24 significant bits -> float (exponent rebiased by 1023 - 127 = 896)
  const float hi = __uint_as_float(sign | __funnelshift_l(ul, mag - (896u << 20), 3));
  // the 29 bits below: an integer times 2^(e - 1075), here 2^-52 2^(e - 1023)
  // with the second factor infinite from e = 1151 (2^128) on
  const float scale = __uint_as_float(sign | ((unsigned int)__vimin_s32_relu(e - 896, 255) << 23));
  const float lo = (__uint2float_rn(ul & 0x1FFFFFFFu) * 0x1p-52f) * scale;
  const bool tiny = e < 1023 - 100;
  return {tiny ? 0.f : hi, tiny ? 0.f : lo};
}

// 1 / sqrt(x) for x > 0: the FP32 estimate y and one correction from the
// residual e = 1 - x y^2 taken in double-float, y (1 + e/2 + 3 e^2/8)
// (Taylor's series of (1 - e)^(-1/2); e is about 1e-7, so the next term is
// below 2^-60).
__device__ __forceinline__ dd dd_rsqrt(dd x) {
  const float y = rsqrtf(x.hi);
  const float q = __fmul_rn(y, y), ql = fmaf(y, y, -q);              // y^2 = q + ql exactly
  const float p = __fmul_rn(x.hi, q);
  const float pl = fmaf(x.hi, ql, fmaf(x.lo, q, fmaf(x.hi, q, -p)));
  const float e = (1.f - p) - pl;
  return dd_fast_two_sum(y, y * (e * fmaf(0.375f, e, 0.5f)));
}

// sqrt(x) for x >= 0: the FP32 root and one Newton correction.
__device__ __forceinline__ dd dd_sqrt(dd x) {
  const float y = sqrtf(x.hi);
  if (!(y > 0.f) || isinf(y)) return {y, 0.f};             // zero, NaN, Inf
  const float r = fmaf(-y, y, x.hi) + x.lo;
  return dd_fast_two_sum(y, r * (0.5f / y));
}

// (out of line, or its FP64 instructions are speculated for every value)
static __device__ __noinline__ double dd_to_double_any(dd x) { return (double)x.hi + (double)x.lo; }

// hi + lo rounded to FP64.  A conversion and an add on the FP64 pipe cost
// three warp instructions of 64 cycles each; this composes the bit pattern
// with integer operations: hi's pattern plus lo as a signed count of units in
// the last place of hi's binade (of the binade below where hi is a power of
// two and lo points towards zero).  Values outside the range where that count
// is an ordinary float go through the conversions.
__device__ __forceinline__ double dd_to_double(dd x) {
  const unsigned int u = __float_as_uint(x.hi);
  const unsigned int e = (u >> 23) & 0xFFu;
  if (e < 56 || e > 254) return dd_to_double_any(x);          // small, zero, Inf, NaN
  const float lo = (u >> 31) ? -x.lo : x.lo;                   // relative to |hi|
  const unsigned int below = (u & 0x7FFFFFu) == 0u && lo < 0.f;
  const int t = __float2int_rn(lo * __uint_as_float((306u + below - e) << 23));
  const unsigned long long m = ((unsigned long long)(e + 896u) << 52) + ((unsigned long long)(u & 0x7FFFFFu) << 29);
  return __longlong_as_double((long long)((m + (long long)t) | ((unsigned long long)(u & 0x80000000u) << 32)));
}

// The FP32 value nearest to x (ties to even) by integer operations on its bit
// pattern -- the top 24 significant bits, rounded on the 29 below -- for x in
// the normal FP32 range; other values go through the conversion instruction.
__device__ __forceinline__ float f32_nearest(double x) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const unsigned int uh = (unsigned int)(u >> 32), ul = (unsigned int)u;
  const int e = (int)((uh >> 20) & 0x7FFu);
  if (e < 897 || e > 1150) return __double2float_rn(x);
  unsigned int f = (uh & 0x80000000u) | ((unsigned int)(e - 896) << 23) | ((uh & 0xFFFFFu) << 3) | (ul >> 29);
  const unsigned int rem = ul & 0x1FFFFFFFu;
  f += (rem > 0x10000000u || (rem == 0x10000000u && (f & 1u))) ? 1u : 0u;
  return __uint_as_float(f);
}

}  // namespace kp
