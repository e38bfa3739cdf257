// Scalar double-float arithmetic: a value is an unevaluated pair of floats (hi, lo),
// hi + lo, with about 48 significant bits.  Products are made error-free with fmaf and
// sums with two-sum, so every operation runs on the FP32 pipes, which GB300 issues at 64
// times its FP64 rate.  Conversions to and from FP64 use integer operations only.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace hbs {

// acc += x * y   (double-float, lazy low part; renormalised by df_norm)
// (explicit _rn intrinsics: the compiler may not contract these into FMAs, which would
// break the error-free transformations)
__device__ __forceinline__ void df_mac(float xh, float xl, float yh, float yl, float& ah, float& al) {
  const float p = __fmul_rn(xh, yh);
  float e = fmaf(xh, yh, -p);
  e = fmaf(xh, yl, e);
  e = fmaf(xl, yh, e);
  const float sum = __fadd_rn(ah, p);
  const float v = __fsub_rn(sum, ah);
  const float t = __fadd_rn(__fsub_rn(ah, __fsub_rn(sum, v)), __fsub_rn(p, v));
  al = __fadd_rn(al, __fadd_rn(t, e));
  ah = sum;
}
__device__ __forceinline__ void df_norm(float& ah, float& al) {
  const float sum = __fadd_rn(ah, al);
  al = __fsub_rn(al, __fsub_rn(sum, ah));
  ah = sum;
}

// Split of an FP64 value into a float pair (hi, lo) without the FP64 conversion path, which
// shares the scarce FP64 pipe: hi carries the top 24 bits of the significand, lo the remainder (29
// bits, an integer conversion) rounded to 24 bits, so hi + lo equals x to 2^-48 relative.
// Values below the float range become 0, values above it infinite.  No branches and no bit
// search: the operands of every double-float product pass through here (with both, the integer
// pipe was 22 % busy beside the multiply-adds of the leaf products).
__device__ __forceinline__ void df_split_bits(double x, float& hi, float& lo) {
  const unsigned int h = (unsigned int)__double2hiint(x), l = (unsigned int)__double2loint(x);
  const unsigned int sgn = h & 0x80000000u, a = h & 0x7FFFFFFFu;
  const bool fits = a >= 0x38100000u && a < 0x47F00000u;  // 2^-126 <= |x| < 2^128
  unsigned int f = __funnelshift_l(l, a - 0x38000000u, 3);  // exponent rebiased by 1023 - 127
  f = fits ? f : (a < 0x38100000u ? 0u : 0x7F800000u);
  // lo = r 2^(e - 1075), r < 2^29: r 2^-29 times 2^(fe - 150), fe the float's exponent field
  const float r = __fmul_rn(__uint2float_rn(l & 0x1FFFFFFFu), 1.862645149230957e-09f);
  const float scale = __uint_as_float((f & 0x7F800000u) - (23u << 23));
  const float v = fits && f >= (24u << 23) ? __fmul_rn(r, scale) : 0.0f;
  hi = __uint_as_float(sgn | f);
  lo = __uint_as_float(sgn | __float_as_uint(v));
}

// float -> double with integer operations only (exact for normal floats; subnormal floats,
// below 1.2e-38, become 0).
__device__ __forceinline__ double f2d_bits(float x) {
  const unsigned int u = __float_as_uint(x);
  const unsigned long long sgn = (unsigned long long)(u & 0x80000000u) << 32;
  const unsigned int e = (u >> 23) & 0xFFu;
  if (e == 0u) return __longlong_as_double((long long)sgn);
  const unsigned long long de = e == 0xFFu ? 0x7FFull : (unsigned long long)(e - 127u + 1023u);
  return __longlong_as_double((long long)(sgn | (de << 52) | ((unsigned long long)(u & 0x7FFFFFu) << 29)));
}

// (ah, al) += (bh, bl), lazy low part.
__device__ __forceinline__ void df_add_to(float bh, float bl, float& ah, float& al) {
  const float sum = __fadd_rn(ah, bh);
  const float v = __fsub_rn(sum, ah);
  const float t = __fadd_rn(__fsub_rn(ah, __fsub_rn(sum, v)), __fsub_rn(bh, v));
  al = __fadd_rn(al, __fadd_rn(t, bl));
  ah = sum;
}

// Double-float square root of a = (ah, al) >= 0: sqrtf of the high part and one Newton
// correction (a - y^2 is exact for y = RN(sqrt(ah)), via fmaf).
__device__ __forceinline__ void df_sqrt(float ah, float al, float& rh, float& rl) {
  if (!(ah > 0.f)) {
    rh = 0.f;
    rl = 0.f;
    return;
  }
  const float y = sqrtf(ah);
  const float e = fmaf(-y, y, ah);
  const float c = __fdiv_rn(__fadd_rn(e, al), __fmul_rn(2.f, y));
  rh = __fadd_rn(y, c);
  rl = __fsub_rn(c, __fsub_rn(rh, y));
}

// Double-float quotient a / b: q1 = ah / bh and one correction from the remainder
// a - q1 b (q1 bh error-free via fmaf).
__device__ __forceinline__ void df_div(float ah, float al, float bh, float bl, float& qh, float& ql) {
  const float q1 = __fdiv_rn(ah, bh);
  const float p = __fmul_rn(q1, bh);
  const float pe = fmaf(q1, bh, -p);
  const float r = __fadd_rn(__fsub_rn(ah, p), __fsub_rn(__fsub_rn(al, pe), __fmul_rn(q1, bl)));
  const float q2 = __fdiv_rn(r, bh);
  qh = __fadd_rn(q1, q2);
  ql = __fsub_rn(q2, __fsub_rn(qh, q1));
}

}  // namespace hbs
