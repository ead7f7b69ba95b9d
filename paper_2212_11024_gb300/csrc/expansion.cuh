// expansion.cuh -- sums of FP32 values carried as unevaluated sums of two or
// three FP32 numbers (error-free transformations: Knuth's TwoSum, Dekker's
// FastTwoSum and the FMA product; Shewchuk 1997, Ogita, Rump and Oishi 2005).
//
// Why: GB300 does 128 FP32 operations per clock and SM but only two FP64
// operations, and a conversion between the two types costs as much as an
// FP64 operation (measured: add, multiply, fma 1.7, F2F 2.0, division 0.22
// per clock and SM).  A sum of FP32 values that an FP64 add would take costs
// 64 FP32 issue slots; the same sum as a three-term expansion costs 13 and
// is more exact (72 bits carried against 53).
#pragma once

#include <cuda_runtime.h>

namespace flame {

struct F2 {  // h + l
  float h, l;
};
struct F3 {  // h + m + l
  float h, m, l;
};

// a + b = h + l exactly.
__device__ __forceinline__ F2 two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float t = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ F2 two_diff(float a, float b) { return two_sum(a, -b); }
// The same for |a| >= |b| (or a = 0).
__device__ __forceinline__ F2 fast_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

__device__ __forceinline__ F2 operator-(F2 a) { return {-a.h, -a.l}; }
__device__ __forceinline__ F3 operator-(F3 a) { return {-a.h, -a.m, -a.l}; }

// Three-term sums; the terms are left unnormalised (each level holds the
// rounding errors of the one above).
__device__ __forceinline__ F3 add3(F2 a, F2 b) {
  const F2 s = two_sum(a.h, b.h), t = two_sum(a.l, b.l), v = two_sum(s.l, t.h);
  return {s.h, v.h, __fadd_rn(t.l, v.l)};
}
__device__ __forceinline__ F3 add3(F3 a, F2 b) {
  const F2 s = two_sum(a.h, b.h), t = two_sum(a.m, b.l), v = two_sum(s.l, t.h);
  return {s.h, v.h, __fadd_rn(a.l, __fadd_rn(t.l, v.l))};
}
__device__ __forceinline__ F3 add3(F3 a, F3 b) {
  const F2 s = two_sum(a.h, b.h), t = two_sum(a.m, b.m), v = two_sum(s.l, t.h);
  return {s.h, v.h, __fadd_rn(__fadd_rn(a.l, b.l), __fadd_rn(t.l, v.l))};
}
__device__ __forceinline__ F3 add3(F2 a, float b) {
  const F2 s = two_sum(a.h, b), t = two_sum(a.l, s.l);
  return {s.h, t.h, t.l};
}
__device__ __forceinline__ F3 add3(F3 a, float b) {
  const F2 s = two_sum(a.h, b), t = two_sum(a.m, s.l);
  return {s.h, t.h, __fadd_rn(a.l, t.l)};
}
// c a power of two
__device__ __forceinline__ F2 scaled(float c, F2 a) { return {c * a.h, c * a.l}; }
__device__ __forceinline__ F3 scaled(float c, F3 a) { return {c * a.h, c * a.m, c * a.l}; }

// Two-term arithmetic (double-float: 48 bits or more), each result
// normalised to |l| <= ulp(h) / 2 where it is passed on to another sum.
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
  const F2 s = two_sum(a.h, b.h);
  return fast_two_sum(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ F2 add2(F2 a, float b) {
  const F2 s = two_sum(a.h, b);
  return fast_two_sum(s.h, __fadd_rn(s.l, a.l));
}
// ... without the normalisation, for a few terms in a row
__device__ __forceinline__ F2 add2u(F2 a, F2 b) {
  const F2 s = two_sum(a.h, b.h);
  return {s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l))};
}
__device__ __forceinline__ F2 add2u(F2 a, float b) {
  const F2 s = two_sum(a.h, b);
  return {s.h, __fadd_rn(s.l, a.l)};
}
__device__ __forceinline__ F2 mul2(float a, float b) {
  const float h = __fmul_rn(a, b);
  return {h, __fmaf_rn(a, b, -h)};
}
__device__ __forceinline__ F2 mul2(float a, F2 b) {
  const float h = __fmul_rn(a, b.h);
  return {h, __fmaf_rn(a, b.l, __fmaf_rn(a, b.h, -h))};
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
  const float h = __fmul_rn(a.h, b.h);
  return {h, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -h)))};
}
// a / b given r = 1 / b.h
__device__ __forceinline__ F2 div2(F2 a, F2 b, float r) {
  const float q = __fmul_rn(a.h, r);
  const float e = __fadd_rn(__fmaf_rn(-q, b.l, __fmaf_rn(-q, b.h, a.h)), a.l);
  return fast_two_sum(q, __fmul_rn(e, r));
}

// An FP32 value as FP64 by its bits (a conversion instruction costs as much
// as an FP64 operation).
__device__ __forceinline__ double widened(float x) {
  const unsigned b = __float_as_uint(x), mag = b & 0x7fffffffu;
  if (mag - 0x00800000u >= 0x7f000000u) return (double)x;  // zero, subnormal or not finite
  return __hiloint2double((int)((mag >> 3) + (896u << 20) | (b & 0x80000000u)), (int)(b << 29));
}

// 1 / d to an FP64 unit or so: two Newton-Raphson steps r += r (1 - d r) on
// the FP32 reciprocal of d's top 24 bits, each doubling its bits (24, 47, 94):
// four FP64 operations, where a division takes about eight times the issue
// slots of one (measured 0.22 a clock and SM against 1.7).  Magnitudes outside
// [2^-100, 2^100] are divided.
__device__ __forceinline__ double reciprocal(double d) {
  const unsigned hi = (unsigned)__double2hiint(d), e = (hi >> 20) & 0x7ffu;
  if (e < 923u || e > 1123u) return 1.0 / d;
  const unsigned top = (((hi & 0x7fffffffu) - (896u << 20)) << 3) | ((unsigned)__double2loint(d) >> 29);
  const double r0 = widened(1.f / __uint_as_float(top | (hi & 0x80000000u)));
  const double r1 = fma(r0, fma(-d, r0, 1.0), r0);
  return fma(r1, fma(-d, r1, 1.0), r1);
}

// An FP64 value as h + l (48 bits or more): h takes the top 24 bits of the
// significand, l the 29 below.  Magnitudes in [2^-74, 2^126) and zero by
// integer operations, others by FP64 instructions.
__device__ __forceinline__ F2 from_double(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x), sign = hi & 0x80000000u;
  const unsigned e = (hi >> 20) & 0x7ffu;
  if (e < 949u || e > 1148u) {
    if (x == 0.0) return {0.f, 0.f};
    const float h = (float)x;
    return {h, (float)(x - (double)h)};
  }
  const unsigned h = (((hi & 0x7fffffffu) - (896u << 20)) << 3) | (lo >> 29);
  const float l = __int2float_rn((int)(lo & 0x1fffffffu)) * __uint_as_float((e - 948u) << 23);
  return {__uint_as_float(h | sign), __uint_as_float(__float_as_uint(l) | sign)};
}

// h + l as FP64, |l| <= ulp(h) / 2, rounded to nearest: the 53-bit result is
// assembled from h's bits and l as an integer in units of its last place, so
// that no FP64 instruction is issued.  Values of h outside [2^-74, 2^127]
// take FP64 instructions.
__device__ __forceinline__ double to_double(F2 a) {
  const unsigned hb = __float_as_uint(a.h), mag = hb & 0x7fffffffu, e = mag >> 23;
  if (mag == 0u) return (double)a.l;
  if (e < 53u || e > 253u) return (double)a.h + (double)a.l;
  // l, signed like h, in units of the last place 2^(exponent(h) - 52), which is
  // half as large below a power of two
  const unsigned lb = __float_as_uint(a.l) ^ (hb & 0x80000000u);
  const bool below = (mag & 0x007fffffu) == 0u && (lb >> 31) != 0u;
  const int n = __float2int_rn(__uint_as_float(lb) * __uint_as_float(((below ? 307u : 306u) - e) << 23));
  const long long bits = ((long long)mag << 29) + (896ll << 52) + n;
  return __longlong_as_double(bits | ((long long)(hb >> 31) << 63));
}
__device__ __forceinline__ double to_double(F3 a) {
  const F2 t = two_sum(a.h, a.m);
  return to_double(two_sum(t.h, __fadd_rn(t.l, a.l)));
}

}  // namespace flame
