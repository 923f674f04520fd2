// Double-float arithmetic for the FP32 pipes.  A value is the unevaluated
// sum hi + lo of two FP32 numbers with |lo| <= ulp(hi) / 2: about 48
// significant bits, with FP32's exponent range.  GB300 issues FP32 FMAs at
// 64 times its FP64 rate, so element passes that need more than FP32 but
// not all of FP64 run several times faster this way.
//
// Built on error-free transformations: TwoSum (Knuth, TAOCP vol. 2,
// Sec. 4.2.2) and FastTwoSum (Dekker 1971) give s + e = a + b exactly;
// TwoProduct with a fused multiply-add gives p + e = a * b exactly.  The
// product is Dekker's double-length multiplication with its cross terms
// folded in by FMA, the quotient long division with two correction steps;
// sums come in Dekker's form (operator+) and an accurate form (both parts
// added separately, renormalised twice) for cancelling totals.
// Requires IEEE FP32 without flush-to-zero and without reassociation (the
// library is built without fast-math).  The products' leading parts are
// __fmul_rn, which the compiler does not contract: an addition fused with the
// multiplication before it would see the exact product, and the error term
// that follows would count its rounding twice.
#pragma once
#include <cuda_runtime.h>

namespace pf {

struct df {
  float hi, lo;
  __host__ __device__ constexpr df() : hi(0.f), lo(0.f) {}
  __host__ __device__ constexpr df(float h, float l) : hi(h), lo(l) {}
  // exact small integers and compile-time constants; a runtime double in
  // device code would cost FP64 instructions (use df_from)
  __host__ __device__ constexpr df(int i) : hi(float(i)), lo(0.f) {}
  __host__ __device__ constexpr df(double d)
      : hi(float(d)), lo(float(d - double(float(d)))) {}
};

__device__ __forceinline__ df df_from(double d) {
  const float h = __double2float_rn(d);
  return df(h, __double2float_rn(d - double(h)));
}
// The same value without FP64 instructions (three conversions and a
// subtraction take the FP64 pipe 64 cycles per warp): the mantissa rounded to
// 24 bits in integer arithmetic, a half up, and the signed rest of at most 28
// bits converted and scaled by a power of two.  Values whose parts leave
// FP32's normal range take the form above.
__device__ __forceinline__ df df_split(double d) {
  const unsigned hw = unsigned(__double2hiint(d)), lw = unsigned(__double2loint(d));
  const unsigned e = (hw >> 20) & 0x7ffu, sign = hw & 0x80000000u;
  if (e - (1023u - 74u) > 74u + 126u) {  // exponent outside [-74, 126]
    if (((hw << 1) | lw) == 0u) return df(__uint_as_float(sign), 0.f);
    return df_from(d);
  }
  const unsigned up = (lw >> 28) & 1u;
  const unsigned h = (((e - 896u) << 23) | ((hw & 0xfffffu) << 3) | (lw >> 29)) + up;
  const float r = float(int(lw & 0x1fffffffu) - int(up << 29));  // times 2^(e - 1023 - 52)
  return df(__uint_as_float(sign | h), r * __uint_as_float(sign | ((e - 948u) << 23)));
}
__device__ __forceinline__ double df_to_double(df x) { return double(x.hi) + double(x.lo); }

// s + e = a + b exactly
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float v = s - a;
  e = (a - (s - v)) + (b - v);
}
// s + e = a + b exactly when |a| >= |b| (or a = 0)
__device__ __forceinline__ void fast_two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  e = b - (s - a);
}

// Accurate double-length sum: error about 2^-47 |x + y| even under
// cancellation.  Used where sums of many elements cancel (nodal sums of
// element contributions, energy totals).
__device__ __forceinline__ df add_accurate(df x, df y) {
  float s, e, t, f;
  two_sum(x.hi, y.hi, s, e);
  two_sum(x.lo, y.lo, t, f);
  e += t;
  fast_two_sum(s, e, s, e);
  e += f;
  fast_two_sum(s, e, s, e);
  return df(s, e);
}

// Dekker's double-length sum: error about 2^-46 (|x| + |y|), half the
// instructions of add_accurate.  The operator form, used inside the element
// algebra, whose intermediate sums do not cancel to far below their terms.
__device__ __forceinline__ df operator+(df x, df y) {
  float s, e;
  two_sum(x.hi, y.hi, s, e);
  e += x.lo + y.lo;
  fast_two_sum(s, e, s, e);
  return df(s, e);
}
__device__ __forceinline__ df operator-(df x) { return df(-x.hi, -x.lo); }
__device__ __forceinline__ df operator-(df x, df y) { return x + (-y); }
__device__ __forceinline__ df operator*(df x, df y) {
  const float p = __fmul_rn(x.hi, y.hi);
  float e = fmaf(x.hi, y.hi, -p);
  e = fmaf(x.hi, y.lo, e);
  e = fmaf(x.lo, y.hi, e);
  float s;
  fast_two_sum(p, e, s, e);
  return df(s, e);
}
__device__ __forceinline__ df operator/(df x, df y) {
  const float q1 = x.hi / y.hi;
  df r = x - y * df(q1, 0.f);
  const float q2 = r.hi / y.hi;
  r = r - y * df(q2, 0.f);
  const float q3 = r.hi / y.hi;
  float s, e;
  fast_two_sum(q1, q2, s, e);
  return df(s, e) + df(q3, 0.f);
}
// x y + z: the product's two parts enter the sum before they are normalised
// (15 FP32 instructions instead of 18)
__device__ __forceinline__ df madd(df x, df y, df z) {
  const float p = __fmul_rn(x.hi, y.hi);
  float e = fmaf(x.hi, y.hi, -p);
  e = fmaf(x.hi, y.lo, e);
  e = fmaf(x.lo, y.hi, e);
  float s, t;
  two_sum(p, z.hi, s, t);
  t += e + z.lo;
  fast_two_sum(s, t, s, t);
  return df(s, t);
}
__device__ __forceinline__ df twice(df x) { return df(2.f * x.hi, 2.f * x.lo); }
__device__ __forceinline__ df& operator+=(df& x, df y) { return x = x + y; }
__device__ __forceinline__ df& operator-=(df& x, df y) { return x = x - y; }
__device__ __forceinline__ df& operator*=(df& x, df y) { return x = x * y; }

}  // namespace pf
