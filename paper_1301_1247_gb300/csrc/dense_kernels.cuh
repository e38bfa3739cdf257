// Batched small dense complex kernels used by the HBS build (Sec. 4): Gauss-Jordan inversion with
// partial pivoting for the per-node blocks, one CTA per matrix, and helpers that the pivoted
// factorizations share.
#pragma once

#include "common.cuh"
#include "dfloat.cuh"
#include "elem.cuh"

namespace hbs {

// Descriptor of one matrix of a batch (pointers into any device buffers, so a batch may
// span several solvers).
struct CpqrJob {
  cplx* mt;    // Mt (m x n, ld = m), overwritten
  cplx* t;     // T output (k x (n - k), ld = k; capacity min(m,n) * n)
  int* perm;   // perm output (n ints)
  int m, n;
  int job;     // index into the rank output array
};

struct InvJob {
  cplx* a;     // matrix (n x n, ld = n), inverted in place
  int n;
  int job;
};

// Block-wide reduction helpers (NT threads, NT multiple of 32).
template <int NT>
__device__ __forceinline__ double block_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < 32) {
    t = threadIdx.x < NT / 32 ? red[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (threadIdx.x == 0) red[0] = t;
  }
  __syncthreads();
  t = red[0];
  __syncthreads();
  return t;
}

// Sum over the block formed in warp 0 alone, so that the other warps issue no FP64
// instructions for it: the values meet in shared memory (red: NT doubles), lane l of
// warp 0 adds those of threads l, l + 32, ... and a butterfly finishes.  The sum is
// returned in every lane of warp 0 (other threads get an unspecified value).  Contains
// one __syncthreads; red may be reused after the caller's next barrier.
template <int NT>
__device__ __forceinline__ double block_sum_warp0(double v, double* red) {
  red[threadIdx.x] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < 32) {
#pragma unroll
    for (int k = 0; k < NT / 32; ++k) t += red[threadIdx.x + 32 * k];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  }
  return t;
}

// Householder reflector H = I - tau v v^H with v = (v0, x_1, x_2, ...) mapping
// x = (x0, x_1, ...) to (beta, 0, ...), beta = -(x0/|x0|) ||x|| (sig = sum_{i>0} |x_i|^2).
__device__ __forceinline__ void householder_scalars(cplx x0, double sig, cplx* v0, cplx* beta, double* tau) {
  const double ax0 = cabs1(x0);
  const double xn = sqrt(ax0 * ax0 + sig);
  const cplx ph = ax0 > 0.0 ? cmk(x0.x / ax0, x0.y / ax0) : cmk(1.0, 0.0);
  *beta = cmk(-ph.x * xn, -ph.y * xn);
  *v0 = csub(x0, *beta);
  const double vv = cabs2(*v0) + sig;
  *tau = vv > 0.0 ? 2.0 / vv : 0.0;
}

// Pivot searches compare squared moduli as IEEE-754 bit patterns read as signed 64-bit
// integers: for non-negative doubles the order is the same, and a -1 marker (an
// eliminated column) sorts below all of them, so the search takes exactly the decisions
// of a floating-point search while leaving the FP64 pipe (1/64 of the FP32 rate on
// GB300; its instructions cost the same with one active lane as with 32) to the updates.
__device__ __forceinline__ long long nkey(double v) { return __double_as_longlong(v); }

__device__ __forceinline__ bool better(long long v, int i, long long bv, int bi) {
  return v > bv || (v == bv && i < bi);
}

constexpr long long kNoKey = (long long)0xBFF0000000000000ull;  // bits of -1.0

// Block-wide (key, index) maximum, lowest index on ties, in every thread.
template <int NT>
__device__ __forceinline__ void block_argmax_key(long long v, int idx, long long* redv, int* redi, long long* outv,
                                                 int* outi) {
  for (int o = 16; o > 0; o >>= 1) {
    const long long v2 = __shfl_xor_sync(0xffffffffu, v, o);
    const int i2 = __shfl_xor_sync(0xffffffffu, idx, o);
    if (better(v2, i2, v, idx)) { v = v2; idx = i2; }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) { redv[warp] = v; redi[warp] = idx; }
  __syncthreads();
  if (threadIdx.x < 32) {
    long long t = threadIdx.x < NT / 32 ? redv[threadIdx.x] : kNoKey;
    int ti = threadIdx.x < NT / 32 ? redi[threadIdx.x] : 0x7fffffff;
    for (int o = 16; o > 0; o >>= 1) {
      const long long t2 = __shfl_xor_sync(0xffffffffu, t, o);
      const int i2 = __shfl_xor_sync(0xffffffffu, ti, o);
      if (better(t2, i2, t, ti)) { t = t2; ti = i2; }
    }
    if (threadIdx.x == 0) { redv[0] = t; redi[0] = ti; }
  }
  __syncthreads();
  *outv = redv[0];
  *outi = redi[0];
  __syncthreads();
}

// Returns (max value, lowest index attaining it) over the block.
template <int NT>
__device__ __forceinline__ void block_argmax(double v, int idx, double* redv, int* redi, double* outv,
                                             int* outi) {
  for (int o = 16; o > 0; o >>= 1) {
    double v2 = __shfl_xor_sync(0xffffffffu, v, o);
    int i2 = __shfl_xor_sync(0xffffffffu, idx, o);
    if (v2 > v || (v2 == v && i2 < idx)) { v = v2; idx = i2; }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) { redv[warp] = v; redi[warp] = idx; }
  __syncthreads();
  if (threadIdx.x < 32) {
    double t = threadIdx.x < NT / 32 ? redv[threadIdx.x] : -1.0;
    int ti = threadIdx.x < NT / 32 ? redi[threadIdx.x] : 0x7fffffff;
    for (int o = 16; o > 0; o >>= 1) {
      double t2 = __shfl_xor_sync(0xffffffffu, t, o);
      int i2 = __shfl_xor_sync(0xffffffffu, ti, o);
      if (t2 > t || (t2 == t && i2 < ti)) { t = t2; ti = i2; }
    }
    if (threadIdx.x == 0) { redv[0] = t; redi[0] = ti; }
  }
  __syncthreads();
  *outv = redv[0];
  *outi = redi[0];
  __syncthreads();
}

// In-place inverse of blocks of n <= kSmallInverse by Gauss-Jordan elimination with partial pivoting, one CTA
// a block, the block in shared memory throughout and nothing interchanged: step c
// exchanges column c with its pivot row p among the rows not taken yet,
//   M(i, j) <- [i != p, j != c] M(i, j) - W(i) P(j),
//   W(i) = M(i, c) / d, W(p) = -1 / d,   P(j) = M(p, j), P(c) = 1,
// and Inv(c, p_t) = M(p_c, t) at the end (as gjx.cu).  W and P are copies, so a step costs two barriers; every
// warp finds the pivot for itself.  The multiply-adds bound it (FP32 pipes in double-float, FP64
// pipe in FP64), with several blocks an SM to cover the barriers.  2048 blocks of 49 in
// double-float: 0.77 ms, and 1.25 with a kernel that streamed the block from L1 and L2 at every step.
constexpr int kSmallInverse = 96;
inline size_t small_inverse_smem(int n) { return (size_t)n * (n + 2) * sizeof(cplx) + (size_t)n * sizeof(int); }

template <typename T>
__global__ void __launch_bounds__(128) k_gj_small(const InvJob* jobs, int* flag_out) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  const InvJob jb = jobs[blockIdx.x];
  const int n = jb.n, tid = threadIdx.x, lane = tid & 31;
  cplx* A = jb.a;
  T* M = reinterpret_cast<T*>(sm_raw);
  T* W = M + n * n;
  T* P = W + n;
  int* perm = reinterpret_cast<int*>(P + n);
  for (int e = tid; e < n * n; e += 128) M[e] = x_in(A[e], (const T*)nullptr);
  const int i0 = tid % n, j0 = tid / n, di = 128 % n, dj = 128 / n;
  unsigned used = 0;  // rows lane, lane + 32, lane + 64
  bool bad = false;
  __syncthreads();
  for (int c = 0; c < n; ++c) {
    unsigned best = 0;
    int bi = 0x7fffffff;
#pragma unroll
    for (int q = 0; q < (kSmallInverse + 31) / 32; ++q) {
      const int i = lane + 32 * q;
      if (i < n && !(used >> q & 1u)) {
        const unsigned k = x_key(M[c * n + i]);
        if (k > best) { best = k; bi = i; }
      }
    }
    const unsigned top = __reduce_max_sync(0xffffffffu, best);
    const int p = __reduce_min_sync(0xffffffffu, best == top ? bi : 0x7fffffff);
    const T d = M[c * n + p];
    const T ip = x_recip(d);
    if (top <= 1u || !x_usable(ip)) {  // the same in every thread
      bad = true;
      break;
    }
    if ((p & 31) == lane) used |= 1u << (p >> 5);
    if (tid < n) {
      W[tid] = tid == p ? x_neg(ip) : x_mul(M[c * n + tid], ip);
      P[tid] = tid == c ? x_in(cmk(1.0, 0.0), (const T*)nullptr) : M[tid * n + p];
    }
    if (tid == 0) perm[c] = p;
    __syncthreads();
    int i = i0, j = j0;
    for (int e = tid; e < n * n; e += 128) {
      T x = (i == p || j == c) ? x_zero<T>() : M[e];
      x_submul(W[i], P[j], x);
      M[e] = x;
      i += di;
      j += dj;
      if (i >= n) {
        i -= n;
        ++j;
      }
    }
    __syncthreads();
  }
  if (!bad) {
    int i = i0, j = j0;
    for (int e = tid; e < n * n; e += 128) {
      A[perm[j] * n + i] = x_out(M[j * n + perm[i]]);
      i += di;
      j += dj;
      if (i >= n) {
        i -= n;
        ++j;
      }
    }
  }
  if (tid == 0) flag_out[jb.job] = bad;
}

}  // namespace hbs
