// Double-float arithmetic: a value is an unevaluated pair of floats (hi, lo), hi + lo,
// with about 48 significant bits.  Products are made error-free with fmaf and sums with
// two-sum, so every operation runs on the FP32 pipes, which GB300 issues at 64 times its
// FP64 rate.  Used for the dense products and the trailing updates of the pivoted QR
// when a handle is built with double-float precision.
#pragma once

#include "common.cuh"
#include "dfcore.cuh"

namespace hbs {

// Complex double-float (16 bytes, the size of a complex double, so a complex128 array
// can hold it in place).
struct __align__(16) dfc {
  float rh, rl, ih, il;
};

__device__ __forceinline__ dfc to_dfc_bits(cplx v) {
  dfc r;
  df_split_bits(v.x, r.rh, r.rl);
  df_split_bits(v.y, r.ih, r.il);
  return r;
}


__device__ __forceinline__ cplx from_dfc_bits(const dfc& v) {
  return cmk(f2d_bits(v.rh) + f2d_bits(v.rl), f2d_bits(v.ih) + f2d_bits(v.il));
}

__device__ __forceinline__ void dfc_norm(dfc& a) {
  df_norm(a.rh, a.rl);
  df_norm(a.ih, a.il);
}

// acc += conj(v) a   (lazy low parts)
__device__ __forceinline__ void dfc_cdot_acc(const dfc& v, const dfc& a, dfc& acc) {
  df_mac(v.rh, v.rl, a.rh, a.rl, acc.rh, acc.rl);
  df_mac(v.ih, v.il, a.ih, a.il, acc.rh, acc.rl);
  df_mac(v.rh, v.rl, a.ih, a.il, acc.ih, acc.il);
  df_mac(-v.ih, -v.il, a.rh, a.rl, acc.ih, acc.il);
}

// a -= v w   (renormalised)
__device__ __forceinline__ void dfc_sub_mul(const dfc& v, const dfc& w, dfc& a) {
  df_mac(-v.rh, -v.rl, w.rh, w.rl, a.rh, a.rl);
  df_mac(v.ih, v.il, w.ih, w.il, a.rh, a.rl);
  df_mac(-v.rh, -v.rl, w.ih, w.il, a.ih, a.il);
  df_mac(-v.ih, -v.il, w.rh, w.rl, a.ih, a.il);
  dfc_norm(a);
}

// a b   (renormalised)
__device__ __forceinline__ dfc dfc_mul(const dfc& a, const dfc& b) {
  dfc r{0.f, 0.f, 0.f, 0.f};
  df_mac(a.rh, a.rl, b.rh, b.rl, r.rh, r.rl);
  df_mac(-a.ih, -a.il, b.ih, b.il, r.rh, r.rl);
  df_mac(a.rh, a.rl, b.ih, b.il, r.ih, r.il);
  df_mac(a.ih, a.il, b.rh, b.rl, r.ih, r.il);
  dfc_norm(r);
  return r;
}

// acc += |a|^2   (lazy low part)
__device__ __forceinline__ void df_abs2_acc(const dfc& a, float& ah, float& al) {
  df_mac(a.rh, a.rl, a.rh, a.rl, ah, al);
  df_mac(a.ih, a.il, a.ih, a.il, ah, al);
}

// s * a for a double-float real s = (sh, sl)   (renormalised)
__device__ __forceinline__ dfc dfc_scale(float sh, float sl, const dfc& a) {
  dfc r{0.f, 0.f, 0.f, 0.f};
  df_mac(sh, sl, a.rh, a.rl, r.rh, r.rl);
  df_mac(sh, sl, a.ih, a.il, r.ih, r.il);
  dfc_norm(r);
  return r;
}

// (h, l) = (ah, al) (bh, bl), and 1 / sqrt(a), 1 / a of a normal a > 0: the FP32 approximation y and
// the first two terms of the series in its residual e (|e| < 2^-21), y (1 + e / 2 + 3 e^2 / 8) and
// y (1 + e + e^2).  A dozen dependent FP32 operations; they sit on the serial chain of every pivot.
__device__ __forceinline__ void df_mul(float ah, float al, float bh, float bl, float& h, float& l) {
  const float p = __fmul_rn(ah, bh);
  float e = fmaf(ah, bh, -p);
  e = fmaf(ah, bl, e);
  e = fmaf(al, bh, e);
  h = __fadd_rn(p, e);
  l = __fsub_rn(e, __fsub_rn(h, p));
}
__device__ __forceinline__ void df_rsqrt(float ah, float al, float& h, float& l) {
  const float y = rsqrtf(ah);
  const float p = __fmul_rn(y, y), pe = fmaf(y, y, -p);
  const float e = __fsub_rn(fmaf(-ah, p, 1.0f), fmaf(ah, pe, __fmul_rn(al, p)));
  const float c = __fmul_rn(y, fmaf(__fmul_rn(e, e), 0.375f, __fmul_rn(e, 0.5f)));
  h = __fadd_rn(y, c);
  l = __fsub_rn(c, __fsub_rn(h, y));
}
__device__ __forceinline__ void df_rcp(float ah, float al, float& h, float& l) {
  float y;
  asm("rcp.approx.f32 %0, %1;" : "=f"(y) : "f"(ah));
  const float e = __fsub_rn(fmaf(-ah, y, 1.0f), __fmul_rn(al, y));
  const float c = __fmul_rn(y, fmaf(e, e, e));
  h = __fadd_rn(y, c);
  l = __fsub_rn(c, __fsub_rn(h, y));
}

// 1 / d = conj(d) / |d|^2 (0 for d = 0)
__device__ __forceinline__ dfc dfc_recip(const dfc& d) {
  float nh = 0.f, nl = 0.f;
  df_abs2_acc(d, nh, nl);
  df_norm(nh, nl);
  if (!(nh > 0.f)) return {0.f, 0.f, 0.f, 0.f};
  float qh, ql;
  df_rcp(nh, nl, qh, ql);
  const dfc c{d.rh, d.rl, -d.ih, -d.il};
  return dfc_scale(qh, ql, c);
}

__device__ __forceinline__ dfc dfc_shfl_xor(const dfc& a, int o) {
  return {__shfl_xor_sync(0xffffffffu, a.rh, o), __shfl_xor_sync(0xffffffffu, a.rl, o),
          __shfl_xor_sync(0xffffffffu, a.ih, o), __shfl_xor_sync(0xffffffffu, a.il, o)};
}

__device__ __forceinline__ dfc dfc_shfl(const dfc& a, int l) {
  return {__shfl_sync(0xffffffffu, a.rh, l), __shfl_sync(0xffffffffu, a.rl, l), __shfl_sync(0xffffffffu, a.ih, l),
          __shfl_sync(0xffffffffu, a.il, l)};
}

// The Householder reflector of x = (x0, x_1, ...) in double-float arithmetic, ||x_1..||^2 = sig: beta =
// -(x0/|x0|) ||x||, v0 = x0 - beta, tau = 2 / (|v0|^2 + sig) = 1 / (||x|| (||x|| + |x0|)).  One thread,
// FP32 pipes only.
__device__ __forceinline__ void df_householder(const dfc& x0, float sh, float sl, dfc* v0, dfc* beta, float* th,
                                               float* tl) {
  float a2h = 0.f, a2l = 0.f;
  df_abs2_acc(x0, a2h, a2l);
  df_norm(a2h, a2l);
  float t2h = a2h, t2l = a2l;
  df_add_to(sh, sl, t2h, t2l);
  df_norm(t2h, t2l);
  if (!(t2h > 1e-36f)) {  // nothing left of the column
    *v0 = *beta = {0.f, 0.f, 0.f, 0.f};
    *th = *tl = 0.f;
    return;
  }
  float rnh, rnl, xnh, xnl;  // 1 / ||x||, ||x||
  df_rsqrt(t2h, t2l, rnh, rnl);
  df_mul(t2h, t2l, rnh, rnl, xnh, xnl);
  // the phase of x0, from x0 2^48 where its square would be too small; none below 2^-108
  const float up = a2h < 1e-24f ? 281474976710656.0f : 1.0f;
  const dfc xs = {x0.rh * up, x0.rl * up, x0.ih * up, x0.il * up};
  float s2h = 0.f, s2l = 0.f;
  df_abs2_acc(xs, s2h, s2l);
  df_norm(s2h, s2l);
  float axh = 0.f, axl = 0.f;
  dfc ph = {1.f, 0.f, 0.f, 0.f};
  if (s2h > 1e-36f) {
    float rah, ral;
    df_rsqrt(s2h, s2l, rah, ral);
    ph = dfc_scale(rah, ral, xs);
    df_mul(s2h, s2l, rah, ral, axh, axl);
    axh /= up;
    axl /= up;
  }
  *beta = dfc_scale(-xnh, -xnl, ph);
  dfc v = x0;
  df_add_to(-beta->rh, -beta->rl, v.rh, v.rl);
  df_add_to(-beta->ih, -beta->il, v.ih, v.il);
  dfc_norm(v);
  *v0 = v;
  float qh = xnh, ql = xnl, ih, il;
  df_add_to(axh, axl, qh, ql);
  df_norm(qh, ql);
  df_rcp(qh, ql, ih, il);
  df_mul(ih, il, rnh, rnl, *th, *tl);
}

// Block-wide double-float sum formed in warp 0 (red: 2 NT floats).  The result is valid
// in every lane of warp 0.  Contains one __syncthreads.
template <int NT>
__device__ __forceinline__ void block_sum_df_warp0(float& h, float& l, float* red) {
  red[threadIdx.x] = h;
  red[NT + threadIdx.x] = l;
  __syncthreads();
  if (threadIdx.x < 32) {
    float sh = 0.f, sl = 0.f;
#pragma unroll
    for (int k = 0; k < NT / 32; ++k) df_add_to(red[threadIdx.x + 32 * k], red[NT + threadIdx.x + 32 * k], sh, sl);
    df_norm(sh, sl);
    for (int o = 16; o > 0; o >>= 1) {
      const float bh = __shfl_xor_sync(0xffffffffu, sh, o), bl = __shfl_xor_sync(0xffffffffu, sl, o);
      df_add_to(bh, bl, sh, sl);
    }
    df_norm(sh, sl);
    h = sh;
    l = sl;
  }
}

// Warp sum of a complex double-float value; every lane receives lane 0's result.
__device__ __forceinline__ dfc dfc_warp_sum(dfc a) {
  dfc_norm(a);
  for (int o = 16; o > 0; o >>= 1) {
    const dfc b = dfc_shfl_xor(a, o);
    df_add_to(b.rh, b.rl, a.rh, a.rl);
    df_add_to(b.ih, b.il, a.ih, a.il);
  }
  dfc_norm(a);
  return dfc_shfl(a, 0);
}

}  // namespace hbs
