// The arithmetic of the factorization kernels for complex FP64 (cplx) and complex double-float (dfc)
// elements under common names, so that one kernel template serves both precisions.
#pragma once

#include "dfloat.cuh"

namespace hbs {

template <typename T> __device__ __forceinline__ T x_zero();
template <> __device__ __forceinline__ cplx x_zero<cplx>() { return cmk(0.0, 0.0); }
template <> __device__ __forceinline__ dfc x_zero<dfc>() { return {0.f, 0.f, 0.f, 0.f}; }
// 1 / d = conj(d) / |d|^2.  FP64: d is scaled by a power of two to a modulus near 1 and 1 / |d|^2
// formed by two Newton steps r <- r (2 - s r) from the FP32 reciprocal (24, 48, then 53 bits), eight
// dependent FP64 operations instead of a complex division's four quotients: the reciprocal is on
// the serial chain of every pivot and an FP64 instruction takes 64 cycles.
__device__ __forceinline__ cplx x_recip(const cplx& d) {
  const int ex = max((__double2hiint(d.x) >> 20) & 0x7ff, (__double2hiint(d.y) >> 20) & 0x7ff);
  if (ex < 64 || ex > 1980) return cabs2(d) > 0.0 ? cdiv(cmk(1.0, 0.0), d) : cmk(0.0, 0.0);
  const double sc = __hiloint2double((2046 - ex) << 20, 0);  // 2^(1023 - ex)
  const double x = d.x * sc, y = d.y * sc;
  const double m = fma(x, x, y * y);  // in [1, 8)
  double r = (double)(1.0f / (float)m);
  r = fma(r, fma(-m, r, 1.0), r);
  r = fma(r, fma(-m, r, 1.0), r);
  r *= sc;
  return cmk(x * r, -y * r);
}
__device__ __forceinline__ dfc x_recip(const dfc& d) { return dfc_recip(d); }
__device__ __forceinline__ cplx x_neg(const cplx& a) { return cmk(-a.x, -a.y); }
__device__ __forceinline__ dfc x_neg(const dfc& a) { return {-a.rh, -a.rl, -a.ih, -a.il}; }
__device__ __forceinline__ cplx x_mul(const cplx& a, const cplx& b) { return cmul(a, b); }
__device__ __forceinline__ dfc x_mul(const dfc& a, const dfc& b) { return dfc_mul(a, b); }
// acc += a b (low parts lazy for dfc; x_norm finishes)
__device__ __forceinline__ void x_mac(const cplx& a, const cplx& b, cplx& acc) { acc = cfma(a, b, acc); }
__device__ __forceinline__ void x_mac(const dfc& a, const dfc& b, dfc& acc) {
  df_mac(a.rh, a.rl, b.rh, b.rl, acc.rh, acc.rl);
  df_mac(-a.ih, -a.il, b.ih, b.il, acc.rh, acc.rl);
  df_mac(a.rh, a.rl, b.ih, b.il, acc.ih, acc.il);
  df_mac(a.ih, a.il, b.rh, b.rl, acc.ih, acc.il);
}
__device__ __forceinline__ void x_norm(cplx&) {}
__device__ __forceinline__ void x_norm(dfc& a) { dfc_norm(a); }
__device__ __forceinline__ cplx x_in(const cplx& v, const cplx*) { return v; }
__device__ __forceinline__ dfc x_in(const cplx& v, const dfc*) { return to_dfc_bits(v); }
__device__ __forceinline__ cplx x_out(const cplx& v) { return v; }
__device__ __forceinline__ cplx x_out(const dfc& v) { return from_dfc_bits(v); }

__device__ __forceinline__ cplx x_shfl(const cplx& v, int l) {
  return cmk(__shfl_sync(0xffffffffu, v.x, l), __shfl_sync(0xffffffffu, v.y, l));
}
__device__ __forceinline__ dfc x_shfl(const dfc& v, int l) { return dfc_shfl(v, l); }

// Pivot keys: |v|^2 to float precision (double-float), or the exponent and upper significand bits of |v|^2
// (FP64), as unsigned integers that order alike; 1 is an exact zero and 0 no candidate.  A square
// carries no sign, so a sign bit belongs to a NaN and is dropped: a key made from it could wrap to 0, and a column
// whose candidates all have key 0 has no pivot row.  A NaN's key is above every number's.  In FP64 the pivot chosen
// is the column's largest to 2^-20 of its square, so that no multiplier passes 1 + 2^-20.
__device__ __forceinline__ unsigned x_key(const cplx& v) {
  const double m = cabs2(v);
  const unsigned hi = (unsigned)__double2hiint(m) & 0x7FFFFFFFu;
  return hi + ((hi | (unsigned)__double2loint(m)) ? 2u : 1u);
}
__device__ __forceinline__ unsigned x_key(const dfc& v) {
  return (__float_as_uint(fmaf(v.rh, v.rh, v.ih * v.ih)) & 0x7FFFFFFFu) + 1u;
}
__device__ __forceinline__ double x_key_value(unsigned k, const cplx*) {
  return k < 2u ? 0.0 : __hiloint2double((int)(k - 2u), k == 2u ? 1 : 0);  // below 2^-1042: some positive value
}
__device__ __forceinline__ double x_key_value(unsigned k, const dfc*) { return (double)__uint_as_float(k - 1u); }
// Whether x_recip found a reciprocal: of a zero, a NaN, an infinity or a value out of the arithmetic's range it
// gives a zero or something not finite, and a block with such a pivot has no inverse.  Integer compares: this
// is beside the serial chain of every pivot.
__device__ __forceinline__ bool x_usable(const cplx& r) {
  const unsigned x = (unsigned)__double2hiint(r.x) & 0x7FFFFFFFu, y = (unsigned)__double2hiint(r.y) & 0x7FFFFFFFu;
  return max(x, y) < 0x7FF00000u && (x | y | (unsigned)__double2loint(r.x) | (unsigned)__double2loint(r.y)) != 0u;
}
__device__ __forceinline__ bool x_usable(const dfc& r) {
  const unsigned x = __float_as_uint(r.rh) & 0x7FFFFFFFu, y = __float_as_uint(r.ih) & 0x7FFFFFFFu;
  return max(x, y) < 0x7F800000u && (x | y) != 0u;
}

// 1 / sqrt(x) of a normal x > 0, and 1 / x of x in [1, 2]: the FP32 value y and a series in its residual e, as a
// float pair good to 2^-44, then one Newton step in FP64.  They sit on a serial chain, where an FP64
// instruction takes 64 cycles: four and three of them instead of ten and six for two Newton steps from FP32.
__device__ __forceinline__ double d_rsqrt(double x) {
  const int e = ((__double2hiint(x) >> 20) & 0x7FF) - 1023, h = e >> 1;  // x = m 4^h, m in [1, 4)
  const double m = __hiloint2double(__double2hiint(x) - (h << 21), __double2loint(x));
  float mh, ml;
  df_split_bits(m, mh, ml);
  const float y = rsqrtf(mh);
  const float p = __fmul_rn(y, y), pe = fmaf(y, y, -p);
  const float r = __fsub_rn(fmaf(-mh, p, 1.0f), fmaf(mh, pe, __fmul_rn(ml, p)));
  const float c = __fmul_rn(y, __fmul_rn(r, fmaf(r, 0.375f, 0.5f)));
  const double d = f2d_bits(y) + f2d_bits(c);  // in (1/2, 1]
  const double half = __hiloint2double(__double2hiint(d) - (1 << 20), __double2loint(d));
  const double q = fma(half, fma(-m, d * d, 1.0), d);
  return __hiloint2double(__double2hiint(q) - (h << 20), __double2loint(q));
}
__device__ __forceinline__ double d_rcp12(double x) {
  float h, l;
  df_split_bits(x, h, l);
  const float y = __frcp_rn(h);
  const float r = __fsub_rn(fmaf(-h, y, 1.0f), __fmul_rn(l, y));
  const double d = f2d_bits(y) + f2d_bits(__fmul_rn(y, fmaf(r, r, r)));
  return fma(d, fma(-x, d, 1.0), d);
}

// Squared norms are FP64 numbers in both arithmetics; a thread's sum of double-float squares is a float pair
// until it joins other threads' sums.
struct dfr {
  float h, l;
};
__device__ __forceinline__ double re_zero(const cplx*) { return 0.0; }
__device__ __forceinline__ dfr re_zero(const dfc*) { return {0.f, 0.f}; }
__device__ __forceinline__ void re_abs2_acc(const cplx& a, double& s) { s = fma(a.x, a.x, fma(a.y, a.y, s)); }
__device__ __forceinline__ void re_abs2_acc(const dfc& a, dfr& s) { df_abs2_acc(a, s.h, s.l); }
__device__ __forceinline__ void re_norm(double&) {}
__device__ __forceinline__ void re_norm(dfr& s) { df_norm(s.h, s.l); }
__device__ __forceinline__ double re_value(double s) { return s; }
__device__ __forceinline__ double re_value(const dfr& s) { return f2d_bits(s.h) + f2d_bits(s.l); }
__device__ __forceinline__ double re_shfl_add(double s, int o) { return s + __shfl_xor_sync(0xffffffffu, s, o); }
// n - |a|^2
__device__ __forceinline__ double re_downdate(double n, const cplx& a) { return n - cabs2(a); }
__device__ __forceinline__ double re_downdate(double n, const dfc& a) {
  float h = 0.f, l = 0.f;
  df_abs2_acc(a, h, l);
  return (n - f2d_bits(h)) - f2d_bits(l);
}
// A real factor in the element's arithmetic.
__device__ __forceinline__ double x_real(double v, const cplx*) { return v; }
__device__ __forceinline__ dfr x_real(double v, const dfc*) {
  dfr r;
  df_split_bits(v, r.h, r.l);
  return r;
}

// acc += conj(v) a (lazy low parts for dfc); a -= v w; s a for a real s
__device__ __forceinline__ void x_cdot(const cplx& v, const cplx& a, cplx& acc) { acc = cfma(cconj(v), a, acc); }
__device__ __forceinline__ void x_cdot(const dfc& v, const dfc& a, dfc& acc) { dfc_cdot_acc(v, a, acc); }
__device__ __forceinline__ void x_submul(const cplx& v, const cplx& w, cplx& a) { a = cfms(v, w, a); }
__device__ __forceinline__ void x_submul(const dfc& v, const dfc& w, dfc& a) { dfc_sub_mul(v, w, a); }
__device__ __forceinline__ cplx x_scale(double s, const cplx& a) { return cscale(a, s); }
__device__ __forceinline__ dfc x_scale(const dfr& s, const dfc& a) { return dfc_scale(s.h, s.l, a); }
// acc += a (lazy low parts for dfc)
__device__ __forceinline__ void x_add(const cplx& a, cplx& acc) { acc = cadd(acc, a); }
__device__ __forceinline__ void x_add(const dfc& a, dfc& acc) {
  df_add_to(a.rh, a.rl, acc.rh, acc.rl);
  df_add_to(a.ih, a.il, acc.ih, acc.il);
}
__device__ __forceinline__ cplx x_shfl_add(const cplx& a, int o) {
  return cmk(a.x + __shfl_xor_sync(0xffffffffu, a.x, o), a.y + __shfl_xor_sync(0xffffffffu, a.y, o));
}
__device__ __forceinline__ dfc x_shfl_add(dfc a, int o) {
  const dfc b = dfc_shfl_xor(a, o);
  df_add_to(b.rh, b.rl, a.rh, a.rl);
  df_add_to(b.ih, b.il, a.ih, a.il);
  return a;
}

// Householder reflector H = I - tau v v^H, v = (v0, x_1, ...), of x = (x0, x_1, ...) with ||x_1..||^2 = sig: beta =
// -(x0 / |x0|) ||x||, v0 = x0 - beta, tau = 2 / (|v0|^2 + sig) = 1 / (||x|| (||x|| + |x0|)).  One warp, in FP64: even
// lanes take ||x|| and real parts, odd lanes |x0| and imaginary parts; the results are in every lane.
__device__ __forceinline__ void warp_householder(const cplx& x0, double sig, int lane, cplx* v0, cplx* beta, double* tau) {
  const bool odd = lane & 1;
  double a2 = cabs2(x0);
  const double t2 = a2 + sig;
  if (!(t2 > 1e-290)) {  // nothing left of the column (the same in every lane)
    *v0 = *beta = cmk(0.0, 0.0);
    *tau = 0.0;
    return;
  }
  double xi = odd ? x0.y : x0.x;
  const double part = xi;
  const bool small = __double2hiint(a2) < 0x05B00000;  // 2^-932: |x0| and the phase from x0 2^400
  if (small) {
    const double up = 0x1p400;
    xi *= up;
    a2 = cabs2(cmk(x0.x * up, x0.y * up));
  }
  const bool phase = a2 > 1e-290;
  const double mine = odd ? (phase ? a2 : 1.0) : t2;
  const double r = d_rsqrt(mine), n = mine * r;  // 1 / ||x||, ||x|| or 1 / |x0|, |x0|
  const double rn = __shfl_sync(0xffffffffu, r, 0), xn = __shfl_sync(0xffffffffu, n, 0);
  const double ra = __shfl_sync(0xffffffffu, r, 1);
  double ax = __shfl_sync(0xffffffffu, n, 1);
  if (small) ax *= 0x1p-400;
  if (!phase) ax = 0.0;
  const double ph = phase ? xi * ra : odd ? 0.0 : 1.0;
  const double b = -(ph * xn), v = part - b;
  *beta = cmk(__shfl_sync(0xffffffffu, b, 0), __shfl_sync(0xffffffffu, b, 1));
  *v0 = cmk(__shfl_sync(0xffffffffu, v, 0), __shfl_sync(0xffffffffu, v, 1));
  *tau = d_rcp12((xn + ax) * rn) * rn * rn;  // xn <= xn + ax <= 2 xn
}

}  // namespace hbs
