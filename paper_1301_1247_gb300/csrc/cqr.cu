// Column-pivoted Householder QR of a tree level's node matrices (the interpolative decompositions
// of Def. 3.1, Sec. 4), each matrix in the shared memory of one cluster of CTAs.
//
// The columns of a matrix (m x n) are dealt to the CS CTAs of its cluster (column j to CTA j mod CS)
// and stay in their shared memory through all steps; a group of GL lanes works on one column
// at a time.  Step s:
//   * the CTAs exchange their best (norm, column) pairs and agree on the pivot column;
//   * every CTA copies rows s.. of it from its owner (distributed shared memory), and one warp forms
//     the reflector (the same arithmetic in every CTA);
//   * every group applies the reflector to its columns, downdates their norms (recomputed on
//     cancellation) and remembers the largest for the next step.
// Columns are never swapped; the permutation kept is the one of the swapping algorithm.  At the
// end R11 and R12 go to global memory, R12 where T is wanted, and k_cqr_tsolve turns it into T =
// R11^{-1} R12.
//
// Norms and the reflector's scalars are FP64 in both arithmetics, products and updates double-float (FP32 pipes)
// on double-float handles.
//
// What bounds it: the chain of a step (two CTA barriers, one cluster barrier, the reflector's scalars:
// about 4 us) for single nodes, the double-float multiply-adds (102 FP32 instructions per element)
// when the level has more matrices than SMs; the matrix is read from HBM or L2 twice.  The kernels it
// replaced streamed every column from L2 at each step (one CTA per matrix, or all SMs with a grid
// barrier per step): the 2048 matrices (65 x 49) and 1024 (90 x 74) of the two lowest levels of a 100 000-node
// build in double-float took 5.5 and 6.4 ms and take 1.9 and 2.9 (1.5 and 2.4 with double-float norms).
//
// The launches are not cooperative: a cluster's CTAs are co-resident by themselves, so a level never
// waits for another thread's persistent kernel.
#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>

#include "dense_kernels.cuh"
#include "elem.cuh"
#include "profile.hpp"
#include "qp_kernels.cuh"

namespace hbs {

namespace {

namespace cg = cooperative_groups;

constexpr int kT = 256;
constexpr int kW = kT / 32;
constexpr size_t kSmemMax = 220 * 1024, kSmemTwo = 110 * 1024;  // one and two CTAs per SM

struct CqrJob {
  const cplx* A;  // m x n, column-major (ld m); read only
  int m, n, kcap;
  int* perm;      // n
  cplx* T;        // k x (n - k)
  cplx* r11;      // k x k, column-major: R11 (upper triangle)
  cplx* invd;     // k: 1 / R_ii
  int* rank;      // rank, and whether it stopped at kcap before the tolerance was met
};

// A squared norm and its column as one integer that orders like (norm, -column): the upper 52 bits and the index
// in the lower 12.  0 for a norm that is not a positive number.  Norms are compared as integers, off the FP64 pipe.
__device__ __forceinline__ unsigned long long c_key(double v, int j) {
  const long long b = __double_as_longlong(v);
  return b > 0 && b <= 0x7FF0000000000000ll ? ((unsigned long long)b & ~0xFFFull) | (4095u - (unsigned)j) : 0ull;
}
__device__ __forceinline__ int c_col(unsigned long long k) { return 4095 - (int)(k & 0xFFFull); }
__device__ __forceinline__ double c_val(unsigned long long k) { return __longlong_as_double((long long)(k & ~0xFFFull)); }
// Cancellation has taken more than 7 of a norm's bits since it was last formed (ref: that norm's 1/128).
__device__ __forceinline__ bool c_cancelled(double t, double ref) {
  return __double_as_longlong(t) <= __double_as_longlong(ref);
}

__device__ __forceinline__ unsigned long long c_warp_max(unsigned long long k) {
  const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(k >> 32));
  const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(k >> 32) == hi ? (unsigned)k : 0u);
  return ((unsigned long long)hi << 32) | lo;
}

// x 2^-e by its exponent field (values that leave the normal range become 0).
__device__ __forceinline__ double c_shift(double x, int e) {
  const int h = __double2hiint(x), ex = ((h >> 20) & 0x7FF) - e;
  return ((h >> 20) & 0x7FF) == 0 || ex < 1 ? 0.0 : __hiloint2double(h - (e << 20), __double2loint(x));
}

// Bytes of shared memory of one CTA.
template <typename T>
__host__ __device__ inline size_t c_smem(int m, int n, int CS) {
  const size_t ncl = (size_t)(n + CS - 1) / CS;
  return 16 * (ncl * m + (CS > 1 ? m : 0) + ncl) + 16 * ncl + 8 * ncl + 8 * (size_t)n + 64;
}

template <typename T, int GL>
__global__ void __launch_bounds__(kT, 2) k_cqr(const CqrJob* jobs, int CS, double tol) {
  using Sum = decltype(re_zero((const T*)nullptr));      // a thread's sum of squares
  using Real = decltype(x_real(0.0, (const T*)nullptr));  // a real factor
  constexpr int G = 32 / GL, NG = kT / GL;
  extern __shared__ __align__(16) unsigned char c_raw[];
  __shared__ unsigned long long s_key[2][8 * kW];  // best of every warp of the cluster, by step parity
  __shared__ T s_v0, s_beta;
  __shared__ Real s_tau;
  __shared__ int s_exp[kW], s_cexp[8], s_nact;
  const CqrJob jb = jobs[blockIdx.x / CS];
  const int rank = (int)blockIdx.x % CS;
  const int m = jb.m, n = jb.n;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, gl = lane % GL, grp = tid / GL;
  const int ncl = n > rank ? (n - rank + CS - 1) / CS : 0, ncap = (n + CS - 1) / CS;
  T* cols = reinterpret_cast<T*>(c_raw);                 // ncap columns of m
  T* vbuf = cols + (size_t)ncap * m;                     // the pivot column (CS > 1)
  T* betac = vbuf + (CS > 1 ? m : 0);                    // R_ss of the columns that were pivots
  double* nrm = reinterpret_cast<double*>(betac + ncap);
  double* ref = nrm + ncap;
  int* elim = reinterpret_cast<int*>(ref + ncap);        // step a column was pivot of, -1 before
  int* act = elim + ncap;                                // the columns that were not pivots, in any order
  int* perm = act + ncap;                                // CTA 0: the permutation and its inverse
  int* pos = perm + n;

  // ---- the matrix, scaled by a power of two to a largest entry near 1 (the squared norms span tol^2)
  int ex = 0;
  for (int64_t e = tid; e < (int64_t)ncl * m; e += kT) {
    const cplx v = jb.A[(int64_t)(rank + CS * (int)(e / m)) * m + e % m];
    ex = max(ex, max((__double2hiint(v.x) >> 20) & 0x7FF, (__double2hiint(v.y) >> 20) & 0x7FF));
  }
  ex = __reduce_max_sync(0xffffffffu, ex);
  if (lane == 0) s_exp[warp] = ex;
  __syncthreads();
  for (int w = 0; w < kW; ++w) ex = max(ex, s_exp[w]);
  if (CS > 1) {
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();  // every CTA has started
    if (tid < CS) *cl.map_shared_rank(&s_cexp[rank], tid) = ex;
    cl.sync();
    for (int q = 0; q < CS; ++q) ex = max(ex, s_cexp[q]);
  }
  const int sh = ex > 0 && ex < 0x7FF ? ex - 1023 : 0;
  unsigned long long best = 0;
  for (int c0 = 0; c0 < ncl; c0 += NG) {
    const int c = c0 + grp;
    double s2 = 0.0;
    if (c < ncl) {
      const cplx* a = jb.A + (int64_t)(rank + CS * c) * m;
      T* d = cols + (size_t)c * m;
      for (int i = gl; i < m; i += GL) {
        const cplx v = a[i];
        const cplx x = cmk(c_shift(v.x, sh), c_shift(v.y, sh));
        d[i] = x_in(x, (const T*)nullptr);
        re_abs2_acc(x, s2);
      }
    }
    for (int o = GL / 2; o > 0; o >>= 1) s2 = re_shfl_add(s2, o);
    if (c < ncl) {
      if (gl == 0) {
        nrm[c] = s2;
        ref[c] = 0.0078125 * s2;
        elim[c] = -1;
        act[c] = c;
      }
      best = max(best, c_key(s2, rank + CS * c));
    }
  }
  if (rank == 0)
    for (int i = tid; i < n; i += kT) perm[i] = pos[i] = i;
  if (tid == 0) s_nact = ncl;

  double thr2 = 0.0;
  int s = 0, capped = 0;
  for (;; ++s) {
    best = c_warp_max(best);
    const int par = s & 1;
    if (CS == 1) {
      if (lane == 0) s_key[par][warp] = best;
      __syncthreads();
    } else {
      cg::cluster_group cl = cg::this_cluster();
      if (lane < CS) *cl.map_shared_rank(&s_key[par][rank * kW + warp], lane) = best;
      cl.sync();
    }
    unsigned long long key = 0;
    for (int q = lane; q < CS * kW; q += 32) key = max(key, s_key[par][q]);
    key = c_warp_max(key);
    const double pv = c_val(key);
    if (s == 0) thr2 = tol * tol * pv;
    const bool met = !(pv > thr2);  // |R_ss| <= tol |R_00|, compared squared; nothing left; not a number
    if (met || s >= jb.kcap) {
      capped = !met && s < min(m, n);
      break;
    }
    const int j = c_col(key), owner = j % CS, jc = j / CS;
    // the pivot column: warp 0 forms the reflector, the others bring the column over meanwhile
    const T* src = CS > 1 ? cg::this_cluster().map_shared_rank(cols, owner) + (size_t)jc * m : cols + (size_t)jc * m;
    const T* v = CS > 1 ? vbuf : src;
    if (warp == 0) {
      Sum part = re_zero((const T*)nullptr);
      const cplx x0 = x_out(src[s]);
#pragma unroll 4
      for (int i = s + 1 + lane; i < m; i += 32) re_abs2_acc(src[i], part);
      double sig = re_value(part);
      for (int o = 16; o > 0; o >>= 1) sig = re_shfl_add(sig, o);
      cplx h0, beta;
      double th;
      warp_householder(x0, sig, lane, &h0, &beta, &th);
      if (lane == 0) {
        s_v0 = x_in(h0, (const T*)nullptr);
        s_tau = x_real(th, (const T*)nullptr);
        s_beta = x_in(beta, (const T*)nullptr);
      }
    } else {
      if (tid == kT - 1) {
        if (rank == owner) {  // out of the active list (nobody reads it between the two barriers)
          elim[jc] = s;
          int q = 0;
          while (act[q] != jc) ++q;
          act[q] = act[--s_nact];
        }
        if (rank == 0) {  // swap the pivot into position s
          const int ps = pos[j];
          if (ps != s) {
            const int cs = perm[s];
            perm[s] = j;
            perm[ps] = cs;
            pos[cs] = ps;
            pos[j] = s;
          }
        }
      }
      if (CS > 1)
        for (int i = s + 1 + tid - 32; i < m; i += kT - 32) vbuf[i] = src[i];
    }
    __syncthreads();
    const T v0 = s_v0;
    const Real tau = s_tau;
    const int nact = s_nact;
    if (tid == 0 && rank == owner) betac[jc] = s_beta;
    best = 0;
    for (int q0 = 0; q0 < nact; q0 += NG) {
      const bool on = q0 + grp < nact;
      const int c = on ? act[q0 + grp] : 0, gj = rank + CS * c;
      if (!__any_sync(0xffffffffu, on)) continue;
      T* a = cols + (size_t)c * m;
      const int end = on ? m : 0;
      T w = x_zero<T>(), w2 = x_zero<T>();  // two chains of sums
      for (int i = s + 1 + gl; i < end; i += 4 * GL) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (i + u * GL < end) x_cdot(v[i + u * GL], a[i + u * GL], u & 1 ? w2 : w);
        x_norm(w);
        x_norm(w2);
      }
      x_add(w2, w);
      const T as = a[s];
#pragma unroll
      for (int o = GL / 2; o > 0; o >>= 1) w = x_shfl_add(w, o);
      x_norm(w);
      x_cdot(v0, as, w);
      x_norm(w);
      w = x_scale(tau, w);
      T top = as;
      x_submul(v0, w, top);
      for (int i = s + 1 + gl; i < end; i += 4 * GL) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (i + u * GL < end) {
            T x = a[i + u * GL];
            x_submul(v[i + u * GL], w, x);
            a[i + u * GL] = x;
          }
      }
      double t = on ? re_downdate(nrm[c], top) : 0.0;
      const bool again = on && c_cancelled(t, ref[c]);
      if (__any_sync(0xffffffffu, again)) {  // cancellation: the norm of rows s + 1.. afresh
        Sum part = re_zero((const T*)nullptr);
        if (again)
          for (int i = s + 1 + gl; i < end; i += GL) {
            re_abs2_acc(a[i], part);
            re_norm(part);
          }
        double q = re_value(part);
        for (int o = GL / 2; o > 0; o >>= 1) q = re_shfl_add(q, o);
        if (again) t = q;
      }
      __syncwarp();
      if (on) {
        if (gl == 0) {
          a[s] = top;
          nrm[c] = t;
          if (again) ref[c] = 0.0078125 * t;
        }
        best = max(best, c_key(t, gj));
      }
    }
  }
  // ---- R11, R12, the permutation and the rank
  const int k = s;
  if (CS > 1) cg::this_cluster().sync();
  else __syncthreads();
  const int* posr = CS > 1 ? cg::this_cluster().map_shared_rank(pos, 0) : pos;
  for (int c = grp; c < ncl; c += NG) {
    const T* a = cols + (size_t)c * m;
    const int l = elim[c];
    if (l >= 0) {
      for (int i = gl; i <= l; i += GL) jb.r11[(int64_t)l * k + i] = x_out(i == l ? betac[c] : a[i]);
      if (gl == 0) jb.invd[l] = cdiv(cmk(1.0, 0.0), x_out(betac[c]));
    } else {
      cplx* t = jb.T + (int64_t)(posr[rank + CS * c] - k) * k;
      for (int i = gl; i < k; i += GL) t[i] = x_out(a[i]);
    }
  }
  if (rank == 0) {
    for (int i = tid; i < n; i += kT) jb.perm[i] = perm[i];
    if (tid == 0) {
      jb.rank[0] = k;
      jb.rank[1] = capped;
    }
  }
  if (CS > 1) cg::this_cluster().sync();  // CTA 0's positions have been read
}

// T = R11^{-1} T in place, one warp per column held in registers (row r in lane r mod 32).
template <int KR>
__global__ void __launch_bounds__(256) k_cqr_tsolve(const CqrJob* jobs) {
  const CqrJob jb = jobs[blockIdx.y];
  const int k = jb.rank[0], nc = jb.n - k;
  if (k <= 0 || nc <= 0) return;
  const int lane = threadIdx.x & 31;
  const int warp = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), nw = (int)((gridDim.x * blockDim.x) >> 5);
  for (int c = warp; c < nc; c += nw) {
    cplx* x = jb.T + (int64_t)c * k;
    cplx w[KR];
#pragma unroll
    for (int q = 0; q < KR; ++q) w[q] = lane + 32 * q < k ? x[lane + 32 * q] : cmk(0.0, 0.0);
#pragma unroll
    for (int qb = KR - 1; qb >= 0; --qb) {
      for (int ii = 31; ii >= 0; --ii) {
        const int i = qb * 32 + ii;
        if (i >= k) continue;
        cplx xi = cmk(__shfl_sync(0xffffffffu, w[qb].x, ii), __shfl_sync(0xffffffffu, w[qb].y, ii));
        xi = cmul(xi, jb.invd[i]);
        if (lane == ii) w[qb] = xi;
        const cplx* ri = jb.r11 + (int64_t)i * k;
#pragma unroll
        for (int q = 0; q <= qb; ++q) {
          const int r = lane + 32 * q;
          if (r < i) w[q] = cfms(ri[r], xi, w[q]);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < KR; ++q)
      if (lane + 32 * q < k) x[lane + 32 * q] = w[q];
  }
}

// Cluster size: the fewest CTAs that leave room for two per SM (a step's multiply-adds run at half the
// rate with one CTA's warps alone), or else eight that have an SM each; 0 if even those do not hold the
// matrix.  Single nodes spread out further, down to 8 columns per CTA.
template <typename T>
int cluster_size(int m, int n, size_t count) {
  if (c_smem<T>(m, n, 8) > kSmemMax) return 0;
  int cs = 1;
  while (cs < 8 && c_smem<T>(m, n, cs) > kSmemTwo) cs *= 2;
  while (cs < 8 && count * cs * 2 <= 304 && n > 8 * cs) cs *= 2;
  return cs;
}

template <typename T, int GL>
void launch_gl(const CqrJob* dj, int nj, size_t sm, int CS, double tol, cudaStream_t s) {
  HBS_CUDA(raise_smem_limit((const void*)k_cqr<T, GL>, std::max<size_t>(sm, 64 * 1024)));
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(nj * CS));
  cfg.blockDim = dim3(kT);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)CS;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  prof::KScope _ks("k_cqr", s);
  HBS_CUDA(cudaLaunchKernelEx(&cfg, k_cqr<T, GL>, dj, CS, tol));
}

// Lanes per column: 8, 16 or 32, so that a CTA's groups (32, 16, 8) have about one column each at the start.
template <typename T>
void launch_cqr(const CqrJob* dj, int nj, size_t sm, int nmax, int CS, double tol, cudaStream_t s) {
  const int cols = (nmax + CS - 1) / CS;
  if (cols > 20) launch_gl<T, 8>(dj, nj, sm, CS, tol, s);
  else if (cols > 10) launch_gl<T, 16>(dj, nj, sm, CS, tol, s);
  else launch_gl<T, 32>(dj, nj, sm, CS, tol, s);
}

// Streams beside the caller's, for launches of one level that do not depend on one another: taken from a
// process-wide pool (per device and priority) and given back when the caller's stream has been made to
// wait for them; work that is still queued then simply runs before the next borrower's.
struct SideStream {
  int dev = 0, prio = 0;
  cudaStream_t s = nullptr;
  cudaEvent_t ev = nullptr;
};
std::mutex g_side_mu;
std::vector<SideStream> g_side;

SideStream side_borrow(cudaStream_t like) {
  SideStream x;
  HBS_CUDA(cudaGetDevice(&x.dev));
  HBS_CUDA(cudaStreamGetPriority(like, &x.prio));
  {
    std::lock_guard<std::mutex> lk(g_side_mu);
    g_side.reserve(16);  // giving back does not allocate
    for (size_t i = 0; i < g_side.size(); ++i)
      if (g_side[i].dev == x.dev && g_side[i].prio == x.prio) {
        x = g_side[i];
        g_side.erase(g_side.begin() + (long)i);
        return x;
      }
  }
  HBS_CUDA(cudaStreamCreateWithPriority(&x.s, cudaStreamNonBlocking, x.prio));
  const cudaError_t e = cudaEventCreateWithFlags(&x.ev, cudaEventDisableTiming);
  if (e != cudaSuccess) {
    cudaStreamDestroy(x.s);
    HBS_CUDA(e);
  }
  return x;
}
void side_return(const SideStream& x) {
  std::lock_guard<std::mutex> lk(g_side_mu);
  if (g_side.size() < 16) {
    g_side.push_back(x);
    return;
  }
  cudaEventDestroy(x.ev);
  cudaStreamDestroy(x.s);  // its queued work still runs
}

}  // namespace

int cqr_cluster(int m, int n, size_t count, bool df) {
  if (n > 4000 || m < 1 || n < 1) return 0;
  return df ? cluster_size<dfc>(m, n, count) : cluster_size<cplx>(m, n, count);
}

std::vector<int> cqr_run(const std::vector<CpqrJob>& js_in, double tol, cudaStream_t s) {
  const int nj = (int)js_in.size();
  std::vector<int> ranks(nj, 0);
  if (nj == 0) return ranks;
  const bool df = gemm_double_float();
  const int cap = injected_rank_cap();  // tests of the HBS_ERR_RANK path
  // the matrices in the order of their cluster sizes, one launch for each size
  std::vector<int> order(nj), size(nj);
  for (int q = 0; q < nj; ++q) {
    order[q] = q;
    size[q] = cqr_cluster(js_in[q].m, js_in[q].n, nj, df);
    if (size[q] == 0) throw Error(HBS_ERR_INTERNAL, "cluster QR: a matrix does not fit");
  }
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return size[a] < size[b]; });
  std::vector<CpqrJob> js(nj);
  int64_t r11 = 0, inv = 0;
  for (int q = 0; q < nj; ++q) {
    js[q] = js_in[order[q]];
    const int64_t k = std::min(js[q].m, js[q].n);
    r11 += k * k;
    inv += k;
  }
  DevBuf<cplx> R(r11), D(inv);
  DevBuf<int> dr(2 * (size_t)nj);
  std::vector<CqrJob> jobs(nj);
  r11 = inv = 0;
  for (int q = 0; q < nj; ++q) {
    const int k = std::min(js[q].m, js[q].n);
    jobs[q] = {js[q].mt, js[q].m, js[q].n, cap > 0 ? std::min(cap, k) : k, js[q].perm, js[q].t, R.get() + r11,
               D.get() + inv, dr.get() + 2 * q};
    r11 += (int64_t)k * k;
    inv += k;
  }
  DevBuf<CqrJob> dj;
  dj.upload(jobs, s);
  // Every class but the last on a side stream, between two events.  Joined whatever happens: the buffers above and
  // the caller's matrices are freed in the order of s, and a launch that fails must not leave the
  // classes before it reading them.
  struct Sides {
    cudaStream_t s;
    std::vector<SideStream> v;
    bool joined = false;
    explicit Sides(cudaStream_t st) : s(st) { v.reserve(8); }
    void join() {
      for (const auto& x : v) {
        HBS_CUDA(cudaEventRecord(x.ev, x.s));
        HBS_CUDA(cudaStreamWaitEvent(s, x.ev, 0));
      }
      joined = true;
    }
    ~Sides() {
      for (const auto& x : v) {
        if (!joined && (cudaEventRecord(x.ev, x.s) != cudaSuccess || cudaStreamWaitEvent(s, x.ev, 0) != cudaSuccess))
          cudaStreamSynchronize(x.s);
        side_return(x);
      }
    }
  } side(s);
  for (int q0 = 0; q0 < nj;) {
    const int CS = size[order[q0]];
    int q1 = q0, nmax = 0;
    size_t sm = 0;
    for (; q1 < nj && size[order[q1]] == CS; ++q1) {
      nmax = std::max(nmax, js[q1].n);
      sm = std::max(sm, df ? c_smem<dfc>(js[q1].m, js[q1].n, CS) : c_smem<cplx>(js[q1].m, js[q1].n, CS));
    }
    cudaStream_t on = s;
    if (q1 < nj) {
      side.v.push_back(side_borrow(s));
      on = side.v.back().s;
      HBS_CUDA(cudaEventRecord(side.v.back().ev, s));
      HBS_CUDA(cudaStreamWaitEvent(on, side.v.back().ev, 0));
    }
    if (df) launch_cqr<dfc>(dj.get() + q0, q1 - q0, sm, nmax, CS, tol, on);
    else launch_cqr<cplx>(dj.get() + q0, q1 - q0, sm, nmax, CS, tol, on);
    q0 = q1;
  }
  side.join();
  HBS_LAUNCH_CHECK("k_cqr");
  const std::vector<int> h = dr.download(s);
  int kmax = 0, ncmax = 0;
  double fl = 0.0, by = 0.0;
  for (int q = 0; q < nj; ++q) {
    ranks[order[q]] = h[2 * q];
    if (h[2 * q + 1]) throw Error(HBS_ERR_RANK, "interpolative decomposition rank exceeds the supported maximum");
    kmax = std::max(kmax, h[2 * q]);
    ncmax = std::max(ncmax, js[q].n - h[2 * q]);
    const double m = js[q].m, n = js[q].n, k = h[2 * q];
    fl += 8.0 * m * n * k;
    by += 16.0 * m * n + 16.0 * k * (n - k) + 4.0 * n;
  }
  prof::add_work("k_cqr", fl, by);
  if (kmax > 0 && ncmax > 0) {
    prof::KScope _ks("k_cqr_tsolve", s);
    const unsigned bx = (unsigned)std::max(1, std::min(1216 / nj + 1, (ncmax + kW - 1) / kW));
    for (int j0 = 0; j0 < nj; j0 += 65535) {
      const dim3 grid(bx, (unsigned)std::min(65535, nj - j0));
      const CqrJob* p = dj.get() + j0;
      switch ((kmax + 31) / 32) {
        case 1: k_cqr_tsolve<1><<<grid, 256, 0, s>>>(p); break;
        case 2: k_cqr_tsolve<2><<<grid, 256, 0, s>>>(p); break;
        case 3: k_cqr_tsolve<3><<<grid, 256, 0, s>>>(p); break;
        case 4: k_cqr_tsolve<4><<<grid, 256, 0, s>>>(p); break;
        case 5: case 6: k_cqr_tsolve<6><<<grid, 256, 0, s>>>(p); break;
        case 7: case 8: k_cqr_tsolve<8><<<grid, 256, 0, s>>>(p); break;
        default: k_cqr_tsolve<16><<<grid, 256, 0, s>>>(p); break;
      }
    }
  }
  HBS_LAUNCH_CHECK("k_cqr_tsolve");
  return ranks;
}

}  // namespace hbs
