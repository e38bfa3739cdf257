// Blocked Gauss-Jordan elimination with partial pivoting for batches of dense complex systems:
// inverses of the per-node blocks (Sec. 4, the D_tau^{-1} of Eqs. def_muhD..def_muG) and the
// Schur systems of the Bloch phases (Sec. 3).
//
// The elimination is a sequence of exchanges.  An exchange at pivot (p, c), d = M(p, c), is
//     M(p, c) = 1 / d,   M(p, j) = M(p, j) / d,   M(i, c) = -M(i, c) / d,
//     M(i, j) = M(i, j) - M(i, c) M(p, j) / d           (i != p, j != c),
// and rows are never moved: once every column c has been exchanged with its pivot row p_c, the
// inverse is the permuted copy Inv(c, p_t) = M(p_c, t).  The exchanges of a panel of 16 columns
// involve only the panel itself; with W the exchanged panel and P its 16 pivot rows, every
// other column x becomes
//     x(i) = (i in P ? 0 : x(i)) + sum_k W(i, k) x_old(p_k),
// a product with inner dimension 16.  A right-hand side is one more such column, so the systems
// are solved without a back substitution, and the panels W left in place apply the same
// elimination to a later right-hand side (gjx_apply, the refinement).
//
// One launch per panel.  In launch t
//   * one cluster per matrix forms panel t: it applies update t - 1 to the panel's columns on
//     loading them, runs the 16 exchanges with every row of the panel in the registers of one
//     thread, and stores W;
//   * all other clusters apply update t - 1 to strips of 16 of the remaining columns.
// So the serial pivot chain of panel t runs beside the bulk of update t - 1, and nothing waits on a
// grid barrier.  What bounds it: for few or small matrices the pivot chain (one CTA barrier and
// one cluster barrier per column, plus 15 multiply-adds per row), for many or large ones the
// multiply-adds of the strips (FP32 pipes in double-float, FP64 pipe in FP64).
//
// Measured against the column-at-a-time elimination that it replaced (one grid barrier per column,
// every column streamed through L2 at each): inverses in double-float of 16 blocks of 300 in 1.64
// instead of 2.93 ms, 8 of 850 in 12.8 instead of 38.1, one of 1700 in about 13 instead of 40.5, 128 of
// 250 in 4.6 instead of 20.3; in FP64 one of 1000 in 9.1 instead of 20.7.  The Schur system of one
// Bloch phase (about 430 unknowns, double-float, with its refinement) takes 1.1 instead of 7.8 ms.
#include <cooperative_groups.h>

#include <algorithm>
#include <string>
#include <type_traits>

#include "dense_kernels.cuh"
#include "elem.cuh"
#include "gjx.hpp"
#include "profile.hpp"
#include "qp_kernels.cuh"
#include "tune.hpp"

namespace hbs {

namespace {

namespace cg = cooperative_groups;

constexpr int kT = 256;    // threads per CTA
constexpr int kW = kT / 32;
constexpr int kTile = 64;  // rows of a strip's tile
constexpr int kS = 16;     // columns of a strip

__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool ok) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  const int bytes = ok ? 16 : 0;  // 0: the destination is zero-filled and nothing is read
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// A CTA's pivot candidate of one step, as it is sent to every CTA of the cluster: the row's values
// (thread h of a row holds the columns h, h + TPR, ...: TPR runs of B / TPR values), 1 / pivot,
// the pivot's key and its row.
template <typename T, int B>
struct __align__(16) Cand {
  T row[B];
  T ip;
  unsigned key;
  int prow;
  int pad[2];
};

template <typename T, int B>
struct PanelSmem {
  T X[B][B];               // update t - 1: the previous pivot rows' values in this panel's columns
  Cand<T, B> cand[2][8];   // candidates of the cluster's CTAs, by step parity (one CTA: [0][0])
  Cand<T, B> mine;
  unsigned wkey[kW];
  int pprev[B];
};
template <typename T, int B>
struct StripSmem {
  T X[B][kS];
  T W[2][B][kTile];
  int pprev[B];
};

template <typename T>
__device__ __forceinline__ T* x_col(const GjxMat& mt, int j) {
  return j < mt.n ? reinterpret_cast<T*>(mt.A) + (int64_t)j * mt.n
                  : reinterpret_cast<T*>(mt.B) + (int64_t)(j - mt.n) * mt.n;
}

// Rows of a cluster's CTA: `chunk` consecutive ones each.
__device__ __forceinline__ int x_chunk(int n, int CS) { return (((n + CS - 1) / CS) + 31) & ~31; }

// Panel t of one matrix: the rows of CTA `rank`, TPR threads per row (thread h holds columns h, h +
// TPR, ... of the panel, C of them) and RPT rows per thread.
template <typename T, int B, int TPR, int RPT>
__device__ __forceinline__ void gjx_panel(const GjxMat& mt, int t, int CS, int rank, PanelSmem<T, B>& sm) {
  constexpr int C = B / TPR, RW = 32 / TPR;  // columns per thread, rows per warp
  const int n = mt.n, c0 = t * B, nb = min(B, n - c0);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int h = lane / RW, rl = lane % RW;
  const int chunk = x_chunk(n, CS);
  const int r0 = rank * chunk, r1 = min(n, r0 + chunk);
  T a[RPT][C];
  int row[RPT];
  bool cand[RPT];
#pragma unroll
  for (int q = 0; q < RPT; ++q) {
    row[q] = r0 + q * (kT / TPR) + warp * RW + rl;
    const bool ok = row[q] < r1;
    cand[q] = ok && mt.colof[row[q]] < 0;
    if (!ok) row[q] = -1;
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const int j = c * TPR + h;
      a[q][c] = (ok && j < nb) ? x_col<T>(mt, c0 + j)[row[q]] : x_zero<T>();
    }
  }
  if (t > 0) {
    const int cp = c0 - B;
    if (tid < B) sm.pprev[tid] = mt.piv[cp + tid];
    if (tid < B * B) {
      const int kk = tid / B, j = tid % B;
      sm.X[kk][(j % TPR) * C + j / TPR] = j < nb ? x_col<T>(mt, c0 + j)[mt.piv[cp + kk]] : x_zero<T>();
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
      bool isp = false;
#pragma unroll
      for (int kk = 0; kk < B; ++kk) isp |= sm.pprev[kk] == row[q];
      if (isp) {
#pragma unroll
        for (int c = 0; c < C; ++c) a[q][c] = x_zero<T>();
      }
      if (row[q] >= 0) {
        const T* wr = reinterpret_cast<const T*>(mt.A) + (int64_t)cp * n + row[q];
        T w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = wr[(int64_t)i * n];
#pragma unroll 1
        for (int k4 = 0; k4 < B; k4 += 4) {
          T wn[4];  // the next four, in flight during the multiply-adds
          const int kn = k4 + 4 < B ? k4 + 4 : 0;
#pragma unroll
          for (int i = 0; i < 4; ++i) wn[i] = wr[(int64_t)(kn + i) * n];
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int c = 0; c < C; ++c) {
              x_mac(w[i], sm.X[k4 + i][h * C + c], a[q][c]);
              x_norm(a[q][c]);
            }
#pragma unroll
          for (int i = 0; i < 4; ++i) w[i] = wn[i];
        }
      }
    }
  }
  // every CTA of the cluster has started (it may be written to) and has read the panel
  if (CS > 1) cg::this_cluster().sync();
  // The exchanges.  The registers rotate: the column of step s is slot 0 of the threads h = s mod
  // TPR, and their finished column moves to their last slot, so that one loop body serves
  // every step.  In double-float every thread forms the reciprocal of its own candidate, beside the
  // multiply-adds, so that it is not on the chain between the two barriers.
  constexpr bool kOwnRecip = std::is_same<T, dfc>::value;
#pragma unroll 1
  for (int s = 0; s < nb; ++s) {
    const int ho = s % TPR;
    unsigned key = 0;
    int kq = 0;
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
      const unsigned k = cand[q] && h == ho ? x_key(a[q][0]) : 0u;
      if (k > key) { key = k; kq = q; }
    }
    T myip = x_zero<T>();
    if (kOwnRecip) {
#pragma unroll
      for (int q = 0; q < RPT; ++q)
        if (q == kq) myip = x_recip(a[q][0]);
    }
    const unsigned wmax = __reduce_max_sync(0xffffffffu, key);
    const int wl = __ffs(__ballot_sync(0xffffffffu, key == wmax && h == ho)) - 1;
    const int wq = RPT > 1 ? __shfl_sync(0xffffffffu, kq, wl) : 0;
    if (lane == 0) sm.wkey[warp] = wmax;
    __syncthreads();
    const unsigned wk = lane < kW ? sm.wkey[lane] : 0u;
    const unsigned cmax = __reduce_max_sync(0xffffffffu, wk);
    const int ww = __ffs(__ballot_sync(0xffffffffu, lane < kW && wk == cmax)) - 1;
    const int par = CS == 1 ? 0 : (s & 1);
    if (warp == ww) {
      Cand<T, B>& mc = CS == 1 ? sm.cand[0][0] : sm.mine;
      if (rl == wl % RW) {  // the winner's TPR threads
#pragma unroll
        for (int q = 0; q < RPT; ++q)
          if (q == wq) {
#pragma unroll
            for (int c = 0; c < C; ++c) mc.row[h * C + c] = a[q][c];
            if (h == ho) {
              mc.ip = kOwnRecip ? myip : x_recip(a[q][0]);
              mc.prow = row[q];
              mc.key = cmax;
            }
          }
      }
      if (CS > 1) {
        constexpr int kItems = (int)(sizeof(Cand<T, B>) / 16);
        __syncwarp();
        cg::cluster_group cl = cg::this_cluster();
        for (int e = lane; e < kItems * CS; e += 32) {
          const int dst = e / kItems, item = e % kItems;
          Cand<T, B>* rem = cl.map_shared_rank(&sm.cand[par][rank], dst);
          reinterpret_cast<float4*>(rem)[item] = reinterpret_cast<const float4*>(&sm.mine)[item];
        }
      }
    }
    const Cand<T, B>* win = &sm.cand[0][0];
    if (CS == 1) {
      __syncthreads();
    } else {
      cg::this_cluster().sync();
      const unsigned ck = lane < CS ? sm.cand[par][lane & 7].key : 0u;
      const unsigned gmax = __reduce_max_sync(0xffffffffu, ck);
      win = &sm.cand[par][__ffs(__ballot_sync(0xffffffffu, lane < CS && ck == gmax)) - 1];
    }
    const T ip = win->ip;
    const int p = win->prow;
    if (rank == 0 && tid == 0) {
      mt.piv[c0 + s] = p;
      mt.pmag[c0 + s] = x_key_value(win->key, (const T*)nullptr);
      if (win->key <= 1u || !x_usable(ip)) *mt.singular = 1;
    }
    const bool own = h == ho;
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
      const bool isp = row[q] == p;
      T l = isp ? ip : x_neg(x_mul(a[q][0], ip));
      if (TPR > 1) l = x_shfl(l, ho * RW + rl);
      if (isp) {
        cand[q] = false;
        if (own) mt.colof[p] = c0 + s;
      }
      const T* wr = win->row + h * C;
      if (TPR == 1) {
#pragma unroll
        for (int c = 1; c < C; ++c) {
          T v = isp ? x_zero<T>() : a[q][c];
          x_mac(l, wr[c], v);
          x_norm(v);
          a[q][c - 1] = v;
        }
        a[q][C - 1] = l;
      } else {
        T v[C];
#pragma unroll
        for (int c = 0; c < C; ++c) {
          v[c] = isp ? x_zero<T>() : a[q][c];
          x_mac(l, wr[c], v[c]);
          x_norm(v[c]);
        }
#pragma unroll
        for (int c = 0; c < C; ++c) a[q][c] = own ? (c + 1 < C ? v[(c + 1) % C] : l) : v[c];
      }
    }
  }
  const int rot = (nb - h + TPR - 1) / TPR;  // rotations of this thread's slots (C of them: none)
#pragma unroll
  for (int q = 0; q < RPT; ++q) {
    if (row[q] < 0) continue;
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const int j = ((c + rot) % C) * TPR + h;
      if (j < nb) x_col<T>(mt, c0 + j)[row[q]] = a[q][c];
    }
  }
}

// Panel t of a matrix with more rows than eight CTAs hold in registers (4096): every thread walks its rows r0 + tid,
// + kT, ..., and the panel stays where it is, in L2, read and written once a column.  The exchanges are those
// of gjx_panel, the columns in place.  The panel's passes bound it (rows x B x 32 bytes a column over eight SMs), so
// the serial chain weighs more than below 4096; the strips' updates run beside it on all other SMs as there.
// One FP64 system of 4400: 355 ms; an LU on one CTA, at its 8.3 GFLOP/s, would take 27 s.
template <typename T, int B>
__device__ __forceinline__ void gjx_panel_rows(const GjxMat& mt, int t, int CS, int rank, PanelSmem<T, B>& sm) {
  const int n = mt.n, c0 = t * B, nb = min(B, n - c0);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int chunk = x_chunk(n, CS);
  const int r0 = rank * chunk, r1 = min(n, r0 + chunk);
  T* P = reinterpret_cast<T*>(mt.A) + (int64_t)c0 * n;
  cg::cluster_group cl = cg::this_cluster();
  if (t > 0) {
    const int cp = c0 - B;
    if (tid < B) sm.pprev[tid] = mt.piv[cp + tid];
    if (tid < B * B) {
      const int kk = tid / B, j = tid % B;
      sm.X[kk][j] = j < nb ? P[(int64_t)j * n + mt.piv[cp + kk]] : x_zero<T>();
    }
  }
  cl.sync();  // every CTA has started and has read the previous pivot rows
  unsigned key = 0;  // this thread's best candidate for the next column
  int krow = -1;
  for (int i = r0 + tid; i < r1; i += kT) {
    T a[B];
#pragma unroll
    for (int c = 0; c < B; ++c) a[c] = c < nb ? P[(int64_t)c * n + i] : x_zero<T>();
    if (t > 0) {
      bool isp = false;
#pragma unroll
      for (int kk = 0; kk < B; ++kk) isp |= sm.pprev[kk] == i;
      if (isp) {
#pragma unroll
        for (int c = 0; c < B; ++c) a[c] = x_zero<T>();
      }
      const T* wr = P - (int64_t)B * n + i;
#pragma unroll 1
      for (int k = 0; k < B; ++k) {
        const T w = wr[(int64_t)k * n];
#pragma unroll
        for (int c = 0; c < B; ++c) {
          x_mac(w, sm.X[k][c], a[c]);
          x_norm(a[c]);
        }
      }
#pragma unroll
      for (int c = 0; c < B; ++c)
        if (c < nb) P[(int64_t)c * n + i] = a[c];
    }
    const unsigned k = mt.colof[i] < 0 ? x_key(a[0]) : 0u;
    if (k > key) { key = k; krow = i; }
  }
#pragma unroll 1
  for (int s = 0; s < nb; ++s) {
    const unsigned wmax = __reduce_max_sync(0xffffffffu, key);
    const int wl = __ffs(__ballot_sync(0xffffffffu, key == wmax)) - 1;
    if (lane == 0) sm.wkey[warp] = wmax;
    __syncthreads();
    const unsigned wk = lane < kW ? sm.wkey[lane] : 0u;
    const unsigned cmax = __reduce_max_sync(0xffffffffu, wk);
    const int ww = __ffs(__ballot_sync(0xffffffffu, lane < kW && wk == cmax)) - 1;
    const int par = s & 1;
    if (warp == ww) {
      if (lane == wl) {
        sm.mine.key = cmax;
        sm.mine.prow = krow;
        if (cmax > 0) {  // a CTA past the last row has no candidate
#pragma unroll
          for (int c = 0; c < B; ++c) sm.mine.row[c] = c < nb ? P[(int64_t)c * n + krow] : x_zero<T>();
          sm.mine.ip = x_recip(P[(int64_t)s * n + krow]);
        }
      }
      constexpr int kItems = (int)(sizeof(Cand<T, B>) / 16);
      __syncwarp();
      for (int e = lane; e < kItems * CS; e += 32) {
        const int dst = e / kItems, item = e % kItems;
        Cand<T, B>* rem = cl.map_shared_rank(&sm.cand[par][rank], dst);
        reinterpret_cast<float4*>(rem)[item] = reinterpret_cast<const float4*>(&sm.mine)[item];
      }
    }
    cl.sync();
    const unsigned ck = lane < CS ? sm.cand[par][lane & 7].key : 0u;
    const unsigned gmax = __reduce_max_sync(0xffffffffu, ck);
    const Cand<T, B>* win = &sm.cand[par][__ffs(__ballot_sync(0xffffffffu, lane < CS && ck == gmax)) - 1];
    const T ip = win->ip;
    const int p = win->prow;
    if (rank == 0 && tid == 0) {
      mt.piv[c0 + s] = p;
      mt.pmag[c0 + s] = x_key_value(win->key, (const T*)nullptr);
      if (win->key <= 1u || !x_usable(ip)) *mt.singular = 1;
    }
    key = 0;
    krow = -1;
    for (int i = r0 + tid; i < r1; i += kT) {
      T a[B];
#pragma unroll
      for (int c = 0; c < B; ++c) a[c] = c < nb ? P[(int64_t)c * n + i] : x_zero<T>();
      const bool isp = i == p;
      T as = x_zero<T>();
#pragma unroll
      for (int c = 0; c < B; ++c)
        if (c == s) as = a[c];
      const T l = isp ? ip : x_neg(x_mul(as, ip));
      T next = x_zero<T>();
#pragma unroll
      for (int c = 0; c < B; ++c) {
        if (c >= nb) break;
        T v = isp ? x_zero<T>() : a[c];
        x_mac(l, win->row[c], v);
        x_norm(v);
        if (c == s) v = l;
        if (c == s + 1) next = v;
        P[(int64_t)c * n + i] = v;
      }
      if (isp) mt.colof[p] = c0 + s;
      const unsigned k = !isp && mt.colof[i] < 0 ? x_key(next) : 0u;
      if (k > key) { key = k; krow = i; }
    }
  }
}

// Update u on the strip of columns [j0, j0 + 16) that are columns [jlo, jhi) of the system, but for
// those of the panels u and t (skip; a solve's jlo lies past them), the rows of CTA `rank` of the
// cluster.  Every CTA has read the old pivot rows before any of them is written.
template <typename T, int B>
__device__ __forceinline__ void gjx_strip(const GjxMat& mt, int u, int j0, int jlo, int jhi, bool skip, int CS, int rank,
                                          StripSmem<T, B>& sm) {
  const int n = mt.n, cp = u * B;
  const int nk = min(B, n - cp);  // B but for the last panel
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int chunk = x_chunk(n, CS);
  const int r0 = rank * chunk, r1 = min(n, r0 + chunk);
  const T* Wg = reinterpret_cast<const T*>(mt.A) + (int64_t)cp * n;
  auto active = [&](int j) { return j >= jlo && j < jhi && !(skip && j < n && (j / B == u || j / B == u + 1)); };
  auto stage = [&](int buf, int rt) {
#pragma unroll
    for (int i = 0; i < B * kTile / kT; ++i) {
      const int e = tid + kT * i, kk = e / kTile, r = rt + e % kTile;
      const bool ok = kk < nk && r < r1;
      cp_async16(&sm.W[buf][kk][e % kTile], ok ? Wg + (int64_t)kk * n + r : Wg, ok);
    }
    cp_async_commit();
  };
  if (r0 < r1) stage(0, r0);
  if (tid < B) sm.pprev[tid] = tid < nk ? mt.piv[cp + tid] : -1;
  if (tid < B * kS) {
    const int kk = tid / kS, j = j0 + tid % kS;
    sm.X[kk][tid % kS] = (kk < nk && active(j)) ? x_col<T>(mt, j)[mt.piv[cp + kk]] : x_zero<T>();
  }
  if (CS == 1) __syncthreads();
  else cg::this_cluster().sync();
  const int ja = 2 * warp, jb = 2 * warp + 1;
  const bool ca = active(j0 + ja), cb = active(j0 + jb);
  T* xa = ca ? x_col<T>(mt, j0 + ja) : nullptr;
  T* xb = cb ? x_col<T>(mt, j0 + jb) : nullptr;
  int buf = 0;
  for (int rt = r0; rt < r1; rt += kTile) {
    T v[2][2];
    bool ok[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int r = rt + lane + 32 * q;
      ok[q] = r < r1;
      bool keep = ok[q];
#pragma unroll
      for (int kk = 0; kk < B; ++kk) keep &= sm.pprev[kk] != r;
      v[q][0] = (keep && ca) ? xa[r] : x_zero<T>();
      v[q][1] = (keep && cb) ? xb[r] : x_zero<T>();
    }
    if (rt + kTile < r1) {
      stage(buf ^ 1, rt + kTile);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    if (ca || cb) {
#pragma unroll 1
      for (int k4 = 0; k4 < B; k4 += 4) {
#pragma unroll
        for (int kk = k4; kk < k4 + 4; ++kk) {
          const T w0 = sm.W[buf][kk][lane], w1 = sm.W[buf][kk][lane + 32];
          const T x0 = sm.X[kk][ja], x1 = sm.X[kk][jb];
          // renormalised at every term: every fourth left an inverse of 300 with 4.9e-14 of error (3.6e-14 now)
          // for 2 % less time
          x_mac(w0, x0, v[0][0]);
          x_norm(v[0][0]);
          x_mac(w1, x0, v[1][0]);
          x_norm(v[1][0]);
          x_mac(w0, x1, v[0][1]);
          x_norm(v[0][1]);
          x_mac(w1, x1, v[1][1]);
          x_norm(v[1][1]);
        }
      }
#pragma unroll
      for (int q = 0; q < 2; ++q)
        if (ok[q]) {
          const int r = rt + lane + 32 * q;
          if (ca) xa[r] = v[q][0];
          if (cb) xb[r] = v[q][1];
        }
    }
    __syncthreads();  // the buffer just read is staged again for the next tile
    buf ^= 1;
  }
}

// Launch t.  Clusters [0, nm) form panel t of their matrix; cluster nm + m * strips + i applies
// update t - 1 to strip i of matrix m: for an inverse every column but those of the panels t - 1
// and t, for a solve the columns after panel t and the right-hand sides.  The launch may begin
// while its predecessor ends (programmatic dependent launch); nothing is touched before the wait.
template <typename T, int B, int TPR, int RPT>
__global__ void __launch_bounds__(kT, RPT == 1 ? 2 : 1) k_gjx(const GjxMat* mats, int nm, int CS, int t, int strips,
                                                              int invert) {
  __shared__ __align__(16) union Smem {
    __device__ Smem() {}
    PanelSmem<T, B> p;
    StripSmem<T, B> s;
  } sm;
  cudaTriggerProgrammaticLaunchCompletion();
  cudaGridDependencySynchronize();
  const int cl = (int)blockIdx.x / CS, rank = (int)blockIdx.x % CS;
  if (cl < nm) {
    const GjxMat mt = mats[cl];
    if (t * B >= mt.n) return;
    if constexpr (RPT > 0) gjx_panel<T, B, TPR, RPT>(mt, t, CS, rank, sm.p);
    else gjx_panel_rows<T, B>(mt, t, CS, rank, sm.p);
    return;
  }
  const GjxMat mt = mats[(cl - nm) / strips];
  const int i = (cl - nm) % strips, u = t - 1, ns = (mt.n + kS - 1) / kS;
  if (u < 0 || u * B >= mt.n) return;
  if (invert) {
    if (i < ns) gjx_strip<T, B>(mt, u, i * kS, 0, mt.n, true, CS, rank, sm.s);
    return;
  }
  const int jlo = min(mt.n, (t + 1) * B), s0 = jlo < mt.n ? jlo / kS : ns;
  if (s0 + i < ns) {
    gjx_strip<T, B>(mt, u, (s0 + i) * kS, jlo, mt.n, false, CS, rank, sm.s);
  } else {
    const int q0 = (s0 + i - ns) * kS;
    if (q0 < mt.q) gjx_strip<T, B>(mt, u, mt.n + q0, mt.n, mt.n + mt.q, false, CS, rank, sm.s);
  }
}

// The working copies, converted to the working type, and the empty pivot record.
template <typename T>
__global__ void k_gjx_load(const GjxMat* mats, int solve) {
  const GjxMat mt = mats[blockIdx.y];
  const int64_t na = (int64_t)mt.n * mt.n, nb = solve ? (int64_t)mt.n * mt.q : 0;
  const bool copy = mt.A != (void*)mt.srcA;
  T* A = reinterpret_cast<T*>(mt.A);
  T* B = reinterpret_cast<T*>(mt.B);
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < na + nb; e += (int64_t)gridDim.x * blockDim.x) {
    if (e < na) {
      if (copy) A[e] = x_in(mt.srcA[e], (const T*)nullptr);
    } else {
      B[e - na] = x_in(mt.srcB[e - na], (const T*)nullptr);
    }
    if (e < mt.n) mt.colof[e] = -1;
  }
}

// The inverse from the exchanged matrix: Inv(i, j) = M(p_i, column whose pivot row is j).
template <typename T>
__global__ void k_gjx_inverse_out(const GjxMat* mats) {
  const GjxMat mt = mats[blockIdx.y];
  const int n = mt.n;
  const T* A = reinterpret_cast<const T*>(mt.A);
  for (int j = blockIdx.x; j < n; j += gridDim.x) {
    const T* c = A + (int64_t)mt.colof[j] * n;
    for (int i = threadIdx.x; i < n; i += blockDim.x) mt.srcA[(int64_t)j * n + i] = x_out(c[mt.piv[i]]);
  }
}

// The solution x(c) = B(p_c) and the conditioning flag (smallest against largest pivot, or one without a reciprocal).
template <typename T>
__global__ void __launch_bounds__(kT) k_gjx_solution_out(const GjxMat* mats, cplx* const* out, int* illcond) {
  __shared__ double smn[kW], smx[kW];
  const GjxMat mt = mats[blockIdx.x];
  const int n = mt.n;
  cplx* x = out[blockIdx.x];
  for (int j = 0; j < mt.q; ++j) {
    const T* b = reinterpret_cast<const T*>(mt.B) + (int64_t)j * n;
    for (int i = threadIdx.x; i < n; i += kT) x[(int64_t)j * n + i] = x_out(b[mt.piv[i]]);
  }
  double mn = 1e300, mx = 0.0;
  for (int i = threadIdx.x; i < n; i += kT) {
    mn = fmin(mn, mt.pmag[i]);
    mx = fmax(mx, mt.pmag[i]);
  }
  for (int o = 16; o > 0; o >>= 1) {
    mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, o));
    mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  if ((threadIdx.x & 31) == 0) {
    smn[threadIdx.x >> 5] = mn;
    smx[threadIdx.x >> 5] = mx;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kW; ++w) {
      mn = fmin(mn, smn[w]);
      mx = fmax(mx, smx[w]);
    }
    illcond[blockIdx.x] = (mn <= 1e-28 * mx || *mt.singular) ? 1 : 0;
  }
}

// The eliminated matrices' double-float pairs as FP64, in place (the same 16 bytes), for k_gjx_apply.
__global__ void __launch_bounds__(kT) k_gjx_widen(const GjxMat* mats) {
  const GjxMat mt = mats[blockIdx.y];
  const int64_t na = (int64_t)mt.n * mt.n;
  const dfc* d = reinterpret_cast<const dfc*>(mt.A);
  cplx* a = reinterpret_cast<cplx*>(mt.A);
  for (int64_t e = blockIdx.x * (int64_t)kT + threadIdx.x; e < na; e += (int64_t)gridDim.x * kT) {
    const dfc v = d[e];
    a[e] = from_dfc_bits(v);
  }
}

// x += the elimination applied to a residual, in FP64: one cluster of CS CTAs per matrix and QB right-hand sides,
// the rows dealt to its CTAs in chunks, the vectors in their shared memory (two copies, so that a panel costs
// one cluster barrier: a panel reads its pivot rows' values from one copy and writes the other).  Two
// threads a row, real and imaginary part: the FP64 multiply-adds bound it (n^2 of 4 for a right-hand side), and a
// warp instruction keeps its quarter of an SM for 64 cycles.  The first rows' W are on their way
// before the barrier.  One right-hand side of one system of 394: 0.077 ms; ten for each of 100 systems
// 1.45 ms (0.98 at the FP64 pipes' rate), and 0.76 in double-float, which would round the correction to 48 bits.
template <int B, int QB>
__global__ void __launch_bounds__(kT) k_gjx_apply(const GjxMat* mats, int CS, int qblocks, const cplx* const* res,
                                                  cplx* const* out) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double xs[B][QB][2];
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)blockIdx.x % CS, item = (int)blockIdx.x / CS;
  const int m = item / qblocks, j0 = item % qblocks * QB;
  const GjxMat mt = mats[m];
  if (j0 >= mt.q) return;  // the whole cluster
  const int n = mt.n, tid = threadIdx.x, chunk = (n + CS - 1) / CS;
  const int r0 = rank * chunk, rows = max(0, min(chunk, n - r0));
  double* r = reinterpret_cast<double*>(smem_raw);  // [2][chunk][QB][2]
  const int half = chunk * QB * 2;
  const cplx* A = reinterpret_cast<const cplx*>(mt.A);
  for (int e = tid; e < rows * QB; e += kT) {
    const int i = e / QB, j = j0 + e % QB;
    const cplx v = j < mt.q ? res[m][(int64_t)j * n + r0 + i] : cmk(0.0, 0.0);
    r[2 * e] = v.x;
    r[2 * e + 1] = v.y;
  }
  int p = tid < B * QB && tid / QB < n ? mt.piv[tid / QB] : 0;
  int buf = 0;
  for (int c0 = 0; c0 < n; c0 += B, buf ^= 1) {
    const int nk = min(B, n - c0);
    cplx w[B];
    int ci = -1;
    auto load = [&](int e) {
      const cplx* wg = A + (int64_t)c0 * n + r0 + (e >> 1);
#pragma unroll
      for (int k = 0; k < B; ++k) w[k] = k < nk ? wg[(int64_t)k * n] : cmk(0.0, 0.0);
      ci = mt.colof[r0 + (e >> 1)];
    };
    if (tid < 2 * rows) load(tid);
    cl.sync();  // the previous panel's values are there, and its readers of the other copy are done
    if (tid < nk * QB) {
      const double* src = cl.map_shared_rank(r + buf * half, p / chunk) + (p % chunk) * QB * 2 + tid % QB * 2;
      xs[tid / QB][tid % QB][0] = src[0];
      xs[tid / QB][tid % QB][1] = src[1];
    }
    if (tid < B * QB && c0 + B + tid / QB < n) p = mt.piv[c0 + B + tid / QB];
    __syncthreads();
    for (int e = tid; e < 2 * rows; e += kT) {
      if (e != tid) load(e);
      const int part = e & 1, flip = part ? 0 : (int)0x80000000;
      const bool isp = ci >= c0 && ci < c0 + nk;
      const int o = buf * half + (e >> 1) * QB * 2 + part;
      double v[QB];
#pragma unroll
      for (int q = 0; q < QB; ++q) v[q] = isp ? 0.0 : r[o + 2 * q];
#pragma unroll
      for (int k = 0; k < B; ++k) {
        if (k >= nk) break;
        const double wy = __hiloint2double(__double2hiint(w[k].y) ^ flip, __double2loint(w[k].y));  // off the FP64 pipe
#pragma unroll
        for (int q = 0; q < QB; ++q) v[q] = fma(w[k].x, xs[k][q][part], fma(wy, xs[k][q][1 - part], v[q]));
      }
#pragma unroll
      for (int q = 0; q < QB; ++q) r[o + (buf ? -half : half) + 2 * q] = v[q];
    }
    __syncthreads();  // xs
  }
  cl.sync();  // nobody reads another CTA's memory any more
  for (int e = tid; e < rows * QB; e += kT) {
    const int i = e / QB, j = j0 + e % QB;
    if (j >= mt.q) continue;
    cplx* x = out[m] + (int64_t)j * n + mt.colof[r0 + i];
    *x = cadd(*x, cmk(r[buf * half + 2 * e], r[buf * half + 2 * e + 1]));
  }
}

template <typename T, int B, int TPR, int RPT>
void launch_steps(const GjxMat* dm, int nm, int nmax, int qmax, int CS, bool invert, cudaStream_t s) {
  const int np = (nmax + B - 1) / B, ns = (nmax + kS - 1) / kS, qs = (qmax + kS - 1) / kS;
  for (int t = 0; t <= np; ++t) {
    const int strips = t == 0 ? 0 : invert ? ns : std::max(0, ns - ((t + 1) * B) / kS) + qs;
    if (t == np && strips == 0) break;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)((nm + (int64_t)nm * strips) * CS));
    cfg.blockDim = dim3(kT);
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)CS;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    prof::g_launches.fetch_add(1, std::memory_order_relaxed);
    HBS_CUDA(cudaLaunchKernelEx(&cfg, k_gjx<T, B, TPR, RPT>, dm, nm, CS, t, std::max(strips, 1), invert ? 1 : 0));
  }
}

// Panel widths: 16 in double-float; 8 in FP64, where the panel's own multiply-adds (rows x width per
// column, on one cluster's FP64 pipes) weigh more than the launches saved.
template <typename T> struct PanelWidth { static constexpr int value = 16; };
template <> struct PanelWidth<cplx> { static constexpr int value = 8; };

template <typename T>
void launch_any(const GjxMat* dm, int nm, int nmax, int qmax, int CS, bool invert, cudaStream_t s) {
  constexpr int B = PanelWidth<T>::value;
  const int chunk = (((nmax + CS - 1) / CS) + 31) & ~31;  // as x_chunk
  if (4 * chunk <= kT) launch_steps<T, B, 4, 1>(dm, nm, nmax, qmax, CS, invert, s);
  else if (2 * chunk <= kT) launch_steps<T, B, 2, 1>(dm, nm, nmax, qmax, CS, invert, s);
  else if (chunk <= kT) launch_steps<T, B, 1, 1>(dm, nm, nmax, qmax, CS, invert, s);
  else if (chunk <= 2 * kT) launch_steps<T, B, 1, 2>(dm, nm, nmax, qmax, CS, invert, s);
  else launch_steps<T, B, 1, 0>(dm, nm, nmax, qmax, CS, invert, s);  // CS is 8 then (gjx_cluster)
}

}  // namespace

// Default cluster size.  The fewest CTAs that hold a panel's rows one per thread (measured: 250 x 128
// blocks 4.3 ms on one CTA, 4.7 on two; 430 x 8 1.9 ms on two, 2.1 on eight; 850 x 8 12.0 ms on
// four, 13.5 on eight), doubled while more than 64 rows are left per CTA (four threads then share a
// row) and the strips of all matrices do not yet fill the SMs: in double-float 128 CTAs of
// strips (128 x 8: 0.31, 0.30, 0.33 ms on one, two, four CTAs), in FP64, whose panels are slower
// (1/64 of the FP32 rate), 608 (300 x 4: 2.3, 2.0, 1.6 ms on two, four, eight).
int gjx_cluster(int nm, int nmax, bool df) {
  const int64_t strips = (int64_t)nm * ((nmax + kS - 1) / kS);
  int cs = 1;
  while (cs < 8 && (kT * cs < nmax || (nmax > 64 * cs && strips * cs < (df ? 128 : 608)))) cs *= 2;
  return cs;
}

bool gjx_cluster_fits(int cs, int nmax) { return cs == 8 || nmax <= kT * cs; }

void gjx_eliminate(Gjx& g, const std::vector<GjxSys>& sys, bool df, bool invert, int CS, cudaStream_t s) {
  const int nm = (int)sys.size();
  g.nm = nm;
  g.df = df;
  g.nmax = 0;
  g.qmax = 0;
  int64_t rows = 0, ea = 0, eb = 0;
  for (const auto& m : sys) {
    g.nmax = std::max(g.nmax, m.n);
    g.qmax = std::max(g.qmax, m.q);
    rows += m.n;
    ea += (int64_t)m.n * m.n;
    eb += (int64_t)m.n * m.q;
  }
  g.piv.alloc(rows);
  g.colof.alloc(rows);
  g.pmag.alloc(rows);
  g.sing.alloc(nm);
  // an FP64 solve works in place (its matrix is not needed again), everything else on a copy
  const bool in_place = !df && !invert;
  if (!in_place) g.A.alloc(ea);
  g.B.alloc(std::max<int64_t>(eb, 1));
  HBS_CUDA(cudaMemsetAsync(g.sing.get(), 0, sizeof(int) * nm, s));
  std::vector<GjxMat> hm(nm);
  rows = ea = eb = 0;
  for (int i = 0; i < nm; ++i) {
    hm[i] = {in_place ? (void*)sys[i].A : (void*)(g.A.get() + ea), g.B.get() + eb, sys[i].A, sys[i].B, sys[i].n, sys[i].q, g.piv.get() + rows,
             g.colof.get() + rows, g.pmag.get() + rows, g.sing.get() + i};
    rows += sys[i].n;
    ea += (int64_t)sys[i].n * sys[i].n;
    eb += (int64_t)sys[i].n * sys[i].q;
  }
  g.mats.upload(hm, s);
  const GjxMat* dm = g.mats.get();
  const int bx = (int)std::max<int64_t>(1, std::min<int64_t>(((int64_t)g.nmax * (g.nmax + g.qmax) + 1023) / 1024, 1216 / nm + 1));
  if (df) k_gjx_load<dfc><<<dim3(bx, nm), 256, 0, s>>>(dm, invert ? 0 : 1);
  else k_gjx_load<cplx><<<dim3(bx, nm), 256, 0, s>>>(dm, invert ? 0 : 1);
  HBS_LAUNCH_CHECK("k_gjx_load");
  if (df) launch_any<dfc>(dm, nm, g.nmax, g.qmax, CS, invert, s);
  else launch_any<cplx>(dm, nm, g.nmax, g.qmax, CS, invert, s);
  HBS_LAUNCH_CHECK("k_gjx");
}

// In-place inverses of the matrices (pointer, n); throws HBS_WARN_ILLCOND on a singular block.
void gjx_invert(const std::vector<std::pair<cplx*, int>>& mats, cudaStream_t s, const char* what) {
  const bool df = gemm_double_float();
  std::vector<GjxSys> sys;
  int nmax = 0;
  double fl = 0.0;
  for (const auto& m : mats) {
    sys.push_back({m.first, nullptr, m.second, 0});
    nmax = std::max(nmax, m.second);
    fl += 8.0 * (double)m.second * m.second * m.second;
  }
  const int nm = (int)mats.size();
  int n_pow = 1, c_pow = 1;
  while (n_pow < nmax) n_pow *= 2;
  while (c_pow < nm) c_pow *= 2;
  const std::string tkey = "inverse/cluster/n" + std::to_string(n_pow) + "/j" + std::to_string(c_pow) + (df ? "/df" : "");
  const int CS = gjx_tuned_cluster(tkey, nm, nmax, df);
  Gjx g;
  {
    int var = 0;
    while ((1 << var) < CS) ++var;
    tune::Timed timed(tkey, var, 4, s);
    prof::KScope _ks("k_gjx", s, fl, 0.0);
    gjx_eliminate(g, sys, df, true, CS, s);
  }
  {
    prof::KScope _ks("k_gjx_inverse_out", s);
    const dim3 grid(std::max(1, std::min(nmax, 1216 / nm + 1)), nm);
    if (df) k_gjx_inverse_out<dfc><<<grid, 128, 0, s>>>(g.mats.get());
    else k_gjx_inverse_out<cplx><<<grid, 128, 0, s>>>(g.mats.get());
  }
  HBS_LAUNCH_CHECK("k_gjx_inverse_out");
  for (int v : g.sing.download(s))
    if (v) throw Error(HBS_WARN_ILLCOND, std::string("singular block in ") + what);
}

// The cluster size of a shape class: tuned when autotuning is on, else gjx_cluster's.
int gjx_tuned_cluster(const std::string& tkey, int nm, int nmax, bool df) {
  const int def = gjx_cluster(nm, nmax, df);
  int dv = 0;
  while ((1 << dv) < def) ++dv;
  int var = tune::choose(tkey, 4, dv);
  if (!gjx_cluster_fits(1 << var, nmax)) {  // too few rows: not a candidate
    if (tune::exploring(tkey, 4)) tune::record(tkey, var, 4, 1e30f);
    var = dv;
  }
  return 1 << var;
}

void gjx_solution(Gjx& g, cplx* const* out, int* illcond, cudaStream_t s) {
  if (g.df) k_gjx_solution_out<dfc><<<g.nm, kT, 0, s>>>(g.mats.get(), out, illcond);
  else k_gjx_solution_out<cplx><<<g.nm, kT, 0, s>>>(g.mats.get(), out, illcond);
  HBS_LAUNCH_CHECK("k_gjx_solution_out");
}

template <int QB>
static void launch_apply(const Gjx& g, int qblocks, const cplx* const* res, cplx* const* out, cudaStream_t s) {
  // eight CTAs a system until there are eight for every SM, then fewer, whose warps have fewer idle lanes
  int CS = 8;
  const auto smem = [&](int c) { return (size_t)2 * QB * sizeof(cplx) * ((g.nmax + c - 1) / c); };
  while (CS > 1 && (int64_t)g.nm * qblocks * CS > 1216 && smem(CS / 2) <= 48 * 1024) CS /= 2;
  const auto fn = k_gjx_apply<PanelWidth<dfc>::value, QB>;
  HBS_CUDA(raise_smem_limit((const void*)fn, std::max<size_t>(smem(CS), 64 * 1024)));  // static memory counts too
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(g.nm * qblocks * CS));
  cfg.blockDim = dim3(kT);
  cfg.dynamicSmemBytes = smem(CS);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)CS;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  HBS_CUDA(cudaLaunchKernelEx(&cfg, fn, (const GjxMat*)g.mats.get(), CS, qblocks, res, out));
}

void gjx_apply(Gjx& g, const cplx* const* res, cplx* const* out, cudaStream_t s) {
  if (!g.df || g.qmax < 1) throw Error(HBS_ERR_INTERNAL, "elimination: nothing to refine");
  {
    prof::KScope _ks("k_gjx_widen", s);
    const int bx = (int)std::max<int64_t>(1, std::min<int64_t>(((int64_t)g.nmax * g.nmax + 1023) / 1024, 1216 / g.nm + 1));
    k_gjx_widen<<<dim3(bx, g.nm), kT, 0, s>>>(g.mats.get());
  }
  HBS_LAUNCH_CHECK("k_gjx_widen");
  prof::KScope _ks("k_gjx_apply", s);
  // right-hand sides in even blocks of at most five, one at a time where the vectors of five are too long
  const int qblocks = g.nmax > 8 * 1200 ? g.qmax : (g.qmax + 4) / 5;
  switch ((g.qmax + qblocks - 1) / qblocks) {
    case 1: launch_apply<1>(g, qblocks, res, out, s); break;
    case 2: launch_apply<2>(g, qblocks, res, out, s); break;
    case 3: launch_apply<3>(g, qblocks, res, out, s); break;
    case 4: launch_apply<4>(g, qblocks, res, out, s); break;
    default: launch_apply<5>(g, qblocks, res, out, s); break;
  }
  HBS_LAUNCH_CHECK("k_gjx_apply");
}

}  // namespace hbs
