// Batched variable-size complex GEMM: C = alpha * op(A) * B + beta * C for a
// list of jobs of different shapes (one grid, jobs x tiles).  Used for the level-wise
// products of the HBS inversion (Eqs. woodbury, def_muhD..def_muG) and the telescoping
// apply of the compressed inverse (Sec. 4).
#pragma once

#include "common.cuh"
#include "dfloat.cuh"

namespace hbs {

struct GemmJob {
  const cplx* A;
  const cplx* B;
  cplx* C;
  int m, n, k;
  int lda, ldb, ldc;
  cplx alpha, beta;
  int tiles_m, tiles_n;  // ceil(m / BM), ceil(n / BN)
  int tile_base;         // prefix sum of tiles over earlier jobs
  int transA;            // 1: op(A) = A^T (A stored k x m, column-major, leading dimension lda)
  int transC;            // 1: C stored row-major, C(i, j) at C[i ldc + j]
  int a_real_digits = 0; // tensor-core products: 0 for a general A; d > 0 when A is real and each
                         // of its rows needs only its first d digit planes (e.g. 1 for signs)
};

constexpr int GBM = 32, GBN = 32, GBK = 8;

// acc += a b in double-float (re += ar br - ai bi; im += ar bi + ai br), lazy low parts.
__device__ __forceinline__ void dfc_mac_tile(const dfc& a, const dfc& b, dfc& c) {
  df_mac(a.rh, a.rl, b.rh, b.rl, c.rh, c.rl);
  df_mac(-a.ih, -a.il, b.ih, b.il, c.rh, c.rl);
  df_mac(a.rh, a.rl, b.ih, b.il, c.ih, c.il);
  df_mac(a.ih, a.il, b.rh, b.rl, c.ih, c.il);
}

__device__ __forceinline__ void tile_mac(const cplx& a, const cplx& b, cplx& c) { c = cfma(a, b, c); }
__device__ __forceinline__ void tile_mac(const dfc& a, const dfc& b, dfc& c) { dfc_mac_tile(a, b, c); }
__device__ __forceinline__ void tile_norm(cplx&) {}
__device__ __forceinline__ void tile_norm(dfc& c) { dfc_norm(c); }
__device__ __forceinline__ void tile_in(const cplx& v, cplx& o) { o = v; }
__device__ __forceinline__ void tile_in(const cplx& v, dfc& o) { o = to_dfc_bits(v); }
__device__ __forceinline__ cplx tile_out(const cplx& v) { return v; }
__device__ __forceinline__ cplx tile_out(const dfc& v) { return from_dfc_bits(v); }

// The multiply-adds of `kend` values of k for one thread's outputs: rows tr + 8 i, i < R, of one
// column.  The loop is unrolled by 2: fully unrolled (8), the variants' code (48 FP32-pipe
// instructions per complex multiply-add in double-float) overflows the instruction cache and
// the warps stall on instruction fetches; not unrolled at all, the loop overhead shows.
template <int R, typename T>
__device__ __forceinline__ void tile_slice(const T (*As)[GBM + 1], const T (*Bs)[GBN + 1], int tr, int tc, int kend,
                                           T (&acc)[GBM / 8]) {
  if (kend == GBK) {
#pragma unroll 2
    for (int kk = 0; kk < GBK; ++kk) {
      const T b = Bs[kk][tc];
#pragma unroll
      for (int i = 0; i < R; ++i) tile_mac(As[kk][tr + 8 * i], b, acc[i]);
    }
  } else {
#pragma unroll 1
    for (int kk = 0; kk < kend; ++kk) {
      const T b = Bs[kk][tc];
#pragma unroll
      for (int i = 0; i < R; ++i) tile_mac(As[kk][tr + 8 * i], b, acc[i]);
    }
  }
}

// One 32 x 32 output tile per CTA (grid.x = total tiles over all jobs; each CTA finds its job by
// binary search on tile_base).
//
// T = cplx: FP64.  T = dfc: FP64 operands are split on load into float pairs (hi, lo), hi = fl32(x),
// lo = fl32(x - hi), and every multiply-add is carried out in double-float arithmetic on the
// FP32 pipes (error-free product via fmaf, error-free sum via two-sum, about 48 significant
// bits): GB300 issues FP32 FMAs at 64x its FP64 rate, so the double-float product is several
// times faster than DFMA while keeping relative errors near 2^-48 per operation; results are
// written back in FP64.
//
// The arithmetic bounds this kernel, so what it must not do is multiply padding: the level products
// are 35-60 rows, columns or k wide, and a warp instruction costs the same however many of its
// lanes are active.  A warp therefore covers 8 rows x 4 columns, four row groups each: groups of
// 8 rows past m are left out, warps whose 4 columns lie past n skip the arithmetic, and the
// last slice of k ends at K.  (With 16 x 16 threads of 2 x 2 outputs and whole slices, a 690 x 49
// x 49 leaf product executed 1.49 multiply-adds for each that counts; now 1.06.  The transposed
// sweep of N = 10^5 to 690 rows, its double-float products: 37.4 -> 33.7 ms; the apply of a 10^4
// inverse to 192 columns in FP64: 8.4 -> 7.2 ms, 0.94 TFLOP/s of the FP64 pipe's 1.26, edges not counted.)  A loop of
// the double-float multiply-add alone, operands in registers, reaches 5.1 of the 6.7 TFLOP/s that
// its instruction count allows (three-operand FMAs issue at 0.8 per cycle).
//
// Slices are double-buffered in shared memory: while the CTA multiplies one slice, each thread
// already holds its elements of the next in registers (loads issued before the multiply-adds),
// and stores them into the other buffer afterwards, so one barrier per slice suffices and the
// L2 latency of the loads overlaps the arithmetic.
template <typename T>
static __global__ void __launch_bounds__(256, 4) k_zgemm_batched(const GemmJob* jobs, int njobs) {
  __shared__ T As[2][GBK][GBM + 1];
  __shared__ T Bs[2][GBK][GBN + 1];
  int t = blockIdx.x;
  int lo = 0, hi = njobs - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].tile_base <= t) lo = mid; else hi = mid - 1;
  }
  const GemmJob& jb = jobs[lo];
  t -= jb.tile_base;
  const int tm = t % jb.tiles_m, tn = t / jb.tiles_m;
  const int row0 = tm * GBM, col0 = tn * GBN;
  const int tid = threadIdx.x;
  const int tr = tid & 7, tc = tid >> 3;  // warp w: columns 4 w .. 4 w + 3
  T acc[GBM / 8];
#pragma unroll
  for (int i = 0; i < GBM / 8; ++i) tile_in(cmk(0.0, 0.0), acc[i]);
  const int m = jb.m, n = jb.n, K = jb.k;
  const int rg = min(GBM / 8, (m - row0 + 7) / 8);       // row groups of this tile
  const bool live = col0 + (tid >> 5) * 4 < n;           // this warp has columns
  // this thread's element of each slice: A (row ar, slice column ak), B (slice row bk, column bc)
  const bool ta = jb.transA != 0;
  const int ar = ta ? tid >> 3 : tid & 31, ak = ta ? tid & 7 : tid >> 5;
  const int bc = tid >> 3, bk = tid & 7;
  const bool a_row = row0 + ar < m, b_col = col0 + bc < n;
  const cplx* pa = ta ? jb.A + (int64_t)(row0 + ar) * jb.lda + ak : jb.A + (int64_t)ak * jb.lda + row0 + ar;
  const int64_t a_step = ta ? GBK : (int64_t)GBK * jb.lda;
  const cplx* pb = jb.B + (int64_t)(col0 + bc) * jb.ldb + bk;
  cplx av = (a_row && ak < K) ? pa[0] : cmk(0.0, 0.0);
  cplx bv = (b_col && bk < K) ? pb[0] : cmk(0.0, 0.0);
  tile_in(av, As[0][ak][ar]);
  tile_in(bv, Bs[0][bk][bc]);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < K; k0 += GBK) {
    const int k1 = k0 + GBK;
    const bool more = k1 < K;
    if (more) {
      pa += a_step;
      pb += GBK;
      av = (a_row && k1 + ak < K) ? pa[0] : cmk(0.0, 0.0);
      bv = (b_col && k1 + bk < K) ? pb[0] : cmk(0.0, 0.0);
    }
    if (live) {
      const int kend = min(GBK, K - k0);
      if (rg == 4) tile_slice<4>(As[buf], Bs[buf], tr, tc, kend, acc);
      else if (rg == 3) tile_slice<3>(As[buf], Bs[buf], tr, tc, kend, acc);
      else if (rg == 2) tile_slice<2>(As[buf], Bs[buf], tr, tc, kend, acc);
      else tile_slice<1>(As[buf], Bs[buf], tr, tc, kend, acc);
#pragma unroll
      for (int i = 0; i < GBM / 8; ++i) tile_norm(acc[i]);
    }
    if (more) {
      tile_in(av, As[buf ^ 1][ak][ar]);
      tile_in(bv, Bs[buf ^ 1][bk][bc]);
    }
    __syncthreads();
    buf ^= 1;
  }
  const bool unit_alpha = jb.alpha.x == 1.0 && jb.alpha.y == 0.0;
  const bool minus_alpha = jb.alpha.x == -1.0 && jb.alpha.y == 0.0;
  const bool zero_beta = jb.beta.x == 0.0 && jb.beta.y == 0.0;
  const bool unit_beta = jb.beta.x == 1.0 && jb.beta.y == 0.0;
  const int gc = col0 + tc;
#pragma unroll
  for (int i = 0; i < GBM / 8; ++i) {
    const int gr = row0 + tr + 8 * i;
    if (gr < m && gc < n) {
      cplx* c = jb.transC ? jb.C + (int64_t)gr * jb.ldc + gc : jb.C + (int64_t)gc * jb.ldc + gr;
      // the common (alpha, beta) = (1, 0), (1, 1) and (-1, 1) take two or four FP64 adds only
      const cplx sum = tile_out(acc[i]);
      cplx v;
      if (unit_alpha && zero_beta) {
        v = sum;
      } else if (unit_alpha && unit_beta) {
        v = cadd(*c, sum);
      } else if (minus_alpha && unit_beta) {
        v = csub(*c, sum);
      } else {
        v = cmul(jb.alpha, sum);
        if (!zero_beta) v = cfma(jb.beta, *c, v);
      }
      *c = v;
    }
  }
}

// Host helper: fill tile bookkeeping and return the total tile count.
inline int64_t gemm_plan(GemmJob* jobs, int njobs, int bm = GBM, int bn = GBN) {
  int64_t tot = 0;
  for (int i = 0; i < njobs; ++i) {
    jobs[i].tiles_m = (jobs[i].m + bm - 1) / bm;
    jobs[i].tiles_n = (jobs[i].n + bn - 1) / bn;
    if (jobs[i].m <= 0 || jobs[i].n <= 0) { jobs[i].tiles_m = 0; jobs[i].tiles_n = 0; }
    jobs[i].tile_base = (int)tot;
    tot += (int64_t)jobs[i].tiles_m * jobs[i].tiles_n;
  }
  return tot;
}

}  // namespace hbs
