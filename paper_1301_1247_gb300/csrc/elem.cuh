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
// whose candidates all have key 0 has no pivot row.  A NaN's key is above every number's.
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

// r = 1 / sqrt(x) for a normal x > 0: two Newton steps r <- r + r (1 - x r^2) / 2 from the FP32 value, on x
// scaled by a power of four (as x_recip, instead of FP64's long square-root and division chains).
__device__ __forceinline__ double d_rsqrt(double x) {
  const int e = ((__double2hiint(x) >> 20) & 0x7FF) - 1023, h = e >> 1;  // x = m 4^h, m in [1, 4)
  const double m = __hiloint2double(__double2hiint(x) - (h << 21), __double2loint(x));
  double r = (double)rsqrtf((float)m);
  r = fma(0.5 * r, fma(-m, r * r, 1.0), r);
  r = fma(0.5 * r, fma(-m, r * r, 1.0), r);
  return __hiloint2double(__double2hiint(r) - (h << 20), __double2loint(r));
}

// Nonnegative reals (squared norms): double, or a float pair.
struct dfr {
  float h, l;
};
__device__ __forceinline__ double re_zero(const cplx*) { return 0.0; }
__device__ __forceinline__ dfr re_zero(const dfc*) { return {0.f, 0.f}; }
__device__ __forceinline__ void re_abs2_acc(const cplx& a, double& s) { s = fma(a.x, a.x, fma(a.y, a.y, s)); }
__device__ __forceinline__ void re_abs2_acc(const dfc& a, dfr& s) { df_abs2_acc(a, s.h, s.l); }
__device__ __forceinline__ void re_norm(double&) {}
__device__ __forceinline__ void re_norm(dfr& s) { df_norm(s.h, s.l); }
__device__ __forceinline__ double re_shfl_add(double s, int o) { return s + __shfl_xor_sync(0xffffffffu, s, o); }
__device__ __forceinline__ dfr re_shfl_add(dfr s, int o) {
  const float h = __shfl_xor_sync(0xffffffffu, s.h, o), l = __shfl_xor_sync(0xffffffffu, s.l, o);
  df_add_to(h, l, s.h, s.l);
  df_norm(s.h, s.l);
  return s;
}
// n - |a|^2
__device__ __forceinline__ double re_downdate(double n, const cplx& a) { return n - cabs2(a); }
__device__ __forceinline__ dfr re_downdate(dfr n, const dfc& a) {
  float h = 0.f, l = 0.f;
  df_abs2_acc(a, h, l);
  df_norm(h, l);
  df_add_to(-h, -l, n.h, n.l);
  df_norm(n.h, n.l);
  return n;
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

// Householder reflector H = I - tau v v^H, v = (v0, x_1, ...), of x = (x0, x_1, ...) with ||x_1..||^2 = sig:
// beta = -(x0 / |x0|) ||x||, v0 = x0 - beta, tau = 2 / (|v0|^2 + sig) = 1 / (||x|| (||x|| + |x0|)).
__device__ __forceinline__ void x_householder(const cplx& x0, double sig, cplx* v0, cplx* beta, double* tau) {
  const double a2 = cabs2(x0), t2 = a2 + sig;
  if (!(t2 > 1e-290)) {  // nothing left of the column
    *v0 = *beta = cmk(0.0, 0.0);
    *tau = 0.0;
    return;
  }
  const double rn = d_rsqrt(t2), xn = t2 * rn;
  double ax = 0.0;
  cplx ph = cmk(1.0, 0.0);
  if (a2 > 1e-290) {
    const double ra = d_rsqrt(a2);
    ax = a2 * ra;
    ph = cmk(x0.x * ra, x0.y * ra);
  }
  *beta = cmk(-ph.x * xn, -ph.y * xn);
  *v0 = csub(x0, *beta);
  // 1 / (xn + ax), xn <= xn + ax <= 2 xn, by Newton from the FP32 quotient
  const double s = (xn + ax) * rn;  // in [1, 2]
  double r = (double)(1.0f / (float)s);
  r = fma(r, fma(-s, r, 1.0), r);
  r = fma(r, fma(-s, r, 1.0), r);
  *tau = r * rn * rn;
}
__device__ __forceinline__ void x_householder(const dfc& x0, const dfr& sig, dfc* v0, dfc* beta, dfr* tau) {
  df_householder(x0, sig.h, sig.l, v0, beta, &tau->h, &tau->l);
}

}  // namespace hbs
