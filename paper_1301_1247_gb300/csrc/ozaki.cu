// Complex GEMM on the 5th-generation tensor cores (tcgen05) with FP64-class accuracy, by
// splitting the operands into bf16 slices (Ozaki's error-free splitting).
//
// Each row r of op(A) is scaled by 2^-E_r (max |Re|, |Im| < 2^E_r) and each column c of B
// by 2^-E_c, and every real part is written as a 49-bit integer M = sum_i q_i 2^{7(6-i)},
// i = 0..6, with balanced digits: |q_0| <= 128, q_1..q_6 in [-64, 63], small integers that are exact
// in bf16.  A digit product (at most 2^14) is exact in the tensor core, and
//   C_rc = 2^{E_r + E_c - 14} sum_{l=0..6} 2^{-7 l} S_l,   S_l = sum_{i+j=l} sum_k q_i q_j
// (the levels l >= 7 are dropped: together about 2^-48 of max|a| max|b| per product).  Over
// 224 values of k every |S_l| stays below 2 x 224 x (2 x 2^13 + 5 x 2^12) < 2^24, so the FP32
// accumulation in tensor memory is exact; every 224 k the seven level sums are added, as
// integers, to two 64-bit sums per real output (levels 0..3 and 4..6).  Nothing is rounded until the
// sums become one FP64 value at the end.
//
// Per CTA: 128 x 32 outputs; tensor memory holds 7 levels x (re, im) x 32 columns of FP32
// accumulators (level l in columns 32 l and 256 + 32 l).  Shared memory is a ring of three
// stages of 16 k, each with 14 A sub-tiles (re/im x 7 digits, 128 x 16 bf16) and 14 B
// sub-tiles (32 x 16) in the no-swizzle K-major core-matrix layout (8 rows x 16 bytes).  The digit
// planes are stored in HBM in that layout, stage by stage ([tile][stage][k-group][plane][row][8
// k]), so one bulk copy brings a stage's A and another its B, with no tensor map per product (a
// tree level has thousands of products; encoding two maps for each took milliseconds of host
// time).  Since B's digit sub-tiles follow one another, digit i of A meets digits 0..6-i of B in a
// single MMA of N = 32 (7 - i) columns that adds to the levels i..6 at once.
//
// Roles: warp 16 issues the copies, warp 17 the MMAs, warps 0-15 read the accumulators (warp w the rows
// 32 (w mod 4).. and columns 8 (w / 4)..) and write the outputs.  The copies and MMAs of the next
// product run while the outputs of the last are written; only the read of the accumulators
// itself, which fill 448 of tensor memory's 512 columns, stands between two periods.
//
// Per 128 x 32 outputs 4 400 cycles go to reading the accumulators and 8 200 to the FP64 additions that round them
// (22 000 with integer rounding), beside 450 of MMAs for every stage.
//
// What bounds it: the MMAs (28 per 16 k, 3584 columns of N in all) and, within a factor of two, the
// 70 KB that each stage brings from L2.  690 x 192 x 100 000: 2.36 ms, 1.40 PFLOP/s of executed
// bf16 (0.73 of the measured 1.91), against 4.87 ms with a double-float combination of the levels
// every 128 k (as long as the MMAs of the period, and alternating with them) and one thread for
// copies and MMAs; the digit planes 0.84 ms against 3.35 (strided reads, two-byte stores).
#include <algorithm>
#include <cstdint>

#include "dense_kernels.cuh"
#include "dfcore.cuh"
#include "profile.hpp"
#include "qp_kernels.cuh"
#include "zgemm.cuh"

namespace hbs {

namespace {

constexpr int OZ_S = 7;        // digits per operand value
constexpr int OZ_BM = 128;     // rows of C per CTA (tensor-memory lanes)
constexpr int OZ_BN = 32;      // columns of C per CTA
constexpr int OZ_BK = 16;      // k per shared-memory stage (one MMA)
constexpr int OZ_FLUSH = 224;  // k per exact accumulation period
constexpr int OZ_RING = 3;     // stages in flight
constexpr int OZ_NSUB = 2 * OZ_S;                         // sub-tiles per operand and stage
constexpr int OZ_A_PL = OZ_BM * 16;                       // one plane's k-group of A: 128 rows x 16 B
constexpr int OZ_B_PL = OZ_BN * 16;                       // one plane's k-group of B: 32 rows x 16 B
constexpr int OZ_A_ST = 2 * OZ_NSUB * OZ_A_PL;            // a stage of all 14 A planes (56 KB)
constexpr int OZ_B_ST = 2 * OZ_NSUB * OZ_B_PL;            // a stage of all 14 B planes (14 KB)
constexpr int OZ_STAGE = OZ_A_ST + OZ_B_ST;               // 70 KB
constexpr int OZ_SMEM = OZ_RING * OZ_STAGE;               // 210 KB
constexpr int OZ_EPI = 512;                               // threads that read accumulators
constexpr int OZ_EC = 8;                                  // columns each of them holds
constexpr int OZ_NT = OZ_EPI + 64;
constexpr int kZeroRow = -2000;  // exponents up to this: a row of zeros (or of nothing yet)

// One operand of one product: op(X) is rows x K with element (r, k) at X[r ld + k] (trans)
// or X[k ld + r]; its exponents and digit planes go to E and out, the planes stage by stage:
// [row tile][stage of 16 k][k-group of 8][plane][row of the tile][8 k].
struct OzOperand {
  const cplx* X;
  int ld, trans;
  int rows, K, rows_pad, Kpad;
  int tile;     // rows per tile (128 for A, 32 for B)
  int nplanes;  // leading digit planes kept (14; fewer when the rest are known to be zero)
  int* E;
  unsigned short* out;
};

// Exponent E with |x| < 2^E for the value whose FP64 high word is hi.
__device__ __forceinline__ int exp_above(unsigned int hi) {
  const int e = (int)((hi >> 20) & 0x7FFu);
  return e == 0 ? kZeroRow : e - 1022;
}
__device__ __forceinline__ unsigned int abs_hi(const cplx& v) {
  return max((unsigned int)__double2hiint(v.x) & 0x7FFFFFFFu, (unsigned int)__double2hiint(v.y) & 0x7FFFFFFFu);
}

// Row exponents of operand blockIdx.y (E preset to a large negative number): a block takes 32 rows x
// 1024 k, reading along the operand's contiguous direction, and adds its maximum by atomics.
__global__ void __launch_bounds__(256) k_oz_exponents(const OzOperand* ops) {
  __shared__ unsigned int red[8][33];
  const OzOperand op = ops[blockIdx.y];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int KC = 1024;
  const int nrb = (op.rows + 31) / 32, nkc = (op.K + KC - 1) / KC;
  for (int64_t u = blockIdx.x; u < (int64_t)nrb * nkc; u += gridDim.x) {
    const int r0 = (int)(u % nrb) * 32, k0 = (int)(u / nrb) * KC, k1 = min(op.K, k0 + KC);
    if (op.trans) {
      for (int i = 0; i < 4; ++i) {
        const int r = r0 + warp * 4 + i;
        if (r >= op.rows) break;
        const cplx* x = op.X + (int64_t)r * op.ld;
        unsigned int mx = 0;
        for (int k = k0 + lane; k < k1; k += 32) mx = max(mx, abs_hi(x[k]));
        mx = __reduce_max_sync(0xffffffffu, mx);
        if (lane == 0) atomicMax(op.E + r, exp_above(mx));
      }
    } else {
      unsigned int mx = 0;
      const int r = r0 + lane;
      if (r < op.rows) {
        const cplx* x = op.X + r;
#pragma unroll 4
        for (int k = k0 + warp; k < k1; k += 8) mx = max(mx, abs_hi(x[(int64_t)k * op.ld]));
      }
      __syncthreads();  // red's last use
      red[warp][lane] = mx;
      __syncthreads();
      if (warp == 0 && r < op.rows) {
        for (int w = 1; w < 8; ++w) mx = max(mx, red[w][lane]);
        atomicMax(op.E + r, exp_above(mx));
      }
    }
  }
}

// The seven balanced digits of x (row exponent E) as bf16 bits, most significant first, or'ed
// into the 16-bit half `half` of w[0..6].  With 64 added at each of the six lower digit positions the
// digits are the plain 7-bit fields less 64; a field is made a float by its place in the
// significand of 2^23, and a small integer's bf16 is the upper half of its float.
__device__ __forceinline__ void digits_of(double x, int E, int half, unsigned int* w) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7FF);
  long long r = 0;
  if (e != 0 && E > kZeroRow) {
    const unsigned long long mant = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const int sh = 1026 + E - e;  // |M| = round(mant 2^{e - 1075 + 49 - E}) = round(mant >> sh), sh >= 4
    if (sh < 64) r = (long long)((mant + (1ull << (sh - 1))) >> sh);
  }
  if ((long long)b < 0) r = -r;
  r += 0x20408102040ll;  // 64 (1 + 2^7 + ... + 2^35)
  const unsigned int lo = (unsigned int)r, hi = (unsigned int)(r >> 28);  // digits 6..3 and 2..1 below 0
  unsigned int f[OZ_S];
  f[6] = lo & 127u;
  f[5] = (lo >> 7) & 127u;
  f[4] = (lo >> 14) & 127u;
  f[3] = (lo >> 21) & 127u;
  f[2] = hi & 127u;
  f[1] = (hi >> 7) & 127u;
#pragma unroll
  for (int i = 1; i < OZ_S; ++i) {
    const float q = __fsub_rn(__uint_as_float(0x4B000000u | f[i]), 8388672.0f);  // 2^23 + 64
    w[i] = half ? __byte_perm(w[i], __float_as_uint(q), 0x7610) : __float_as_uint(q) >> 16;
  }
  const float q0 = (float)((int)hi >> 14);
  w[0] = half ? __byte_perm(w[0], __float_as_uint(q0), 0x7610) : __float_as_uint(q0) >> 16;
}

// Digit planes of operand blockIdx.y.  One thread per (row, k-group of 8): consecutive threads take
// consecutive rows, so the 16-byte stores of a plane are contiguous, and the reads too unless
// the operand is stored by rows (each thread then reads its own 128 bytes).
__global__ void __launch_bounds__(256) k_oz_digits(const OzOperand* ops) {
  const OzOperand op = ops[blockIdx.y];
  const int64_t tot = (int64_t)op.rows_pad * (op.Kpad / 8);
  const int nkg = op.Kpad / 8;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
    const int row = (int)(e % op.tile);
    const int64_t t = e / op.tile;
    const int kg = (int)(t % nkg), r = (int)(t / nkg) * op.tile + row, k = 8 * kg;
    cplx v[8];
    int E = kZeroRow;
    if (r < op.rows) {
      E = op.E[r];
      const cplx* x = op.trans ? op.X + (int64_t)r * op.ld + k : op.X + (int64_t)k * op.ld + r;
      const int64_t step = op.trans ? 1 : op.ld;
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = k + i < op.K ? x[i * step] : cmk(0.0, 0.0);
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = cmk(0.0, 0.0);
    }
    unsigned short* o = op.out + (t * op.nplanes * op.tile + row) * 8;
#pragma unroll
    for (int part = 0; part < 2; ++part) {
      if (part * OZ_S >= op.nplanes) break;
      unsigned int w[4][OZ_S];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        digits_of(part ? v[2 * i].y : v[2 * i].x, E, 0, w[i]);
        digits_of(part ? v[2 * i + 1].y : v[2 * i + 1].x, E, 1, w[i]);
      }
#pragma unroll
      for (int d = 0; d < OZ_S; ++d)
        if (part * OZ_S + d < op.nplanes)
          *reinterpret_cast<uint4*>(o + (int64_t)(part * OZ_S + d) * op.tile * 8) =
              make_uint4(w[0][d], w[1][d], w[2][d], w[3][d]);
    }
  }
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor: no swizzle, K-major; LBO = the byte offset between the two
// k-adjacent core matrices of a 16-k sub-tile (one k-group region), SBO = 128 B between 8-row
// groups.  The start address sits in the low 14 bits (address / 16), so the descriptor of a
// sub-tile at byte offset o from another is that descriptor plus o / 16.
__device__ __forceinline__ uint64_t oz_desc(uint32_t addr, uint32_t lbo) {
  return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(128 >> 4) << 32) |
         ((uint64_t)1 << 46);
}

// kind::f16 instruction descriptor: D f32, A and B bf16, both K-major, M = 128, N columns.
__host__ __device__ constexpr uint32_t oz_idesc(bool negA, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((negA ? 1u : 0u) << 13) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(OZ_BM >> 4) << 24);
}

__device__ __forceinline__ void oz_mma(uint32_t tmem, uint64_t da, uint64_t db, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(da), "l"(db), "r"(idesc), "r"(acc));
}

// Waits for the mbarrier phase of the given parity; gives up after one second (globaltimer), or
// once another wait of the CTA has given up (*gave_up, which this one then sets too).
__device__ __forceinline__ bool oz_wait(uint32_t bar, uint32_t parity, volatile int* gave_up) {
  uint64_t t0 = 0;
  for (;;) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 1000;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    if (t0 == 0) t0 = t;
    if (*gave_up || t - t0 > 1000000000ull) {
      *gave_up = 1;
      return false;
    }
  }
}

__device__ __forceinline__ void oz_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// Issues the read of 8 accumulator columns (32 lanes); the values are there after tmem_wait().
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
// The registers pass through the wait, so that no use of them can be moved before it.
__device__ __forceinline__ void tmem_wait(uint32_t (&a)[8], uint32_t (&b)[8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]),
                 "+r"(b[0]), "+r"(b[1]), "+r"(b[2]), "+r"(b[3]), "+r"(b[4]), "+r"(b[5]), "+r"(b[6]), "+r"(b[7])
               :
               : "memory");
}

// Bulk copy of `bytes` (a multiple of 16, both addresses 16-byte aligned) into shared memory,
// completing on the mbarrier bar.
__device__ __forceinline__ void oz_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(bar)
               : "memory");
}

// d 2^e: the exponent field moves, or two products (2^e might not be a number) where that leaves the
// normal range.
__device__ __forceinline__ double oz_scale(double d, int e) {
  const int h = __double2hiint(d), x = (h >> 20) & 0x7FF;
  if (x == 0) return d;  // a zero sum
  if (x + e < 1 || x + e > 2046) {
    const int e1 = max(-1000, min(1000, e)), e2 = max(-1000, min(1000, e - e1));
    return d * __hiloint2double((1023 + e1) << 20, 0) * __hiloint2double((1023 + e2) << 20, 0);
  }
  return __hiloint2double(h + (e << 20), __double2loint(d));
}

// A 64-bit integer rounded to FP64, by its halves' places in the significands of 2^84 and 2^52: an FP64
// instruction takes 64 cycles here and an output needs several, so the conversion instructions
// (and the integer pipe: counting zeros and shifting took 22 000 cycles per 128 x 32 outputs) are
// avoided; two additions.
__device__ __forceinline__ double oz_narrow(long long v) {
  const double a = __hiloint2double(0x45300000, (int)((unsigned int)(v >> 32) ^ 0x80000000u));
  const double b = __hiloint2double(0x43300000, (int)(unsigned int)v);
  return __dadd_rn(__dsub_rn(a, __longlong_as_double(0x4530000080100000ll)), b);  // 2^84 + 2^63 + 2^52
}

// hi 2^21 + lo rounded to FP64 once, times 2^e.  width 0: |hi| < 2^41, one 64-bit integer; 1: |hi| < 2^51, each
// part by its place in the significand of 1.5 2^52, two exact subtractions and one multiply-add; 2: any
// hi, the part beyond 64 bits shifted out (|lo| < 2^58).
__device__ __forceinline__ double oz_value(long long hi, long long lo, int e, int width) {
  if (width == 0) return oz_scale(oz_narrow((hi << 21) + lo), e);
  if (width == 1) {
    const double m = 6755399441055744.0;  // 1.5 2^52
    const double a = __dsub_rn(__longlong_as_double(hi + 0x4338000000000000ll), m);
    const double b = __dsub_rn(__longlong_as_double(lo + 0x4338000000000000ll), m);
    return oz_scale(__fma_rn(a, 2097152.0, b), e);
  }
  const int s = max(0, 23 - __clzll(hi ^ (hi >> 63)));  // bits of |hi| beyond 41
  const long long h = s <= 21 ? hi << (21 - s) : hi >> (s - 21);
  return oz_scale(oz_narrow(h + (lo >> s)), e + s);
}

// One product of a batch on the tensor cores.  Work items are (tile_m, tile_n, split);
// item_base is the prefix sum of tiles_m tiles_n splits over the earlier jobs.
struct OzJob {
  const unsigned short* Ad;  // digit planes of op(A) and of B^T, stage by stage
  const unsigned short* Bd;
  const int* Er;
  const int* Ec;
  int m, n, nst, kst, splits, tiles_m, tiles_n;  // stages in all, stages per split
  int nre, nim;  // digit planes of op(A)'s real and imaginary parts that can be nonzero
  int64_t item_base;
  cplx alpha, beta;
  cplx* C;  // splits == 1: C = alpha op(A) B + beta C directly
  int ldc;
  int transC;  // C row-major
  cplx* W;  // splits > 1: alpha (partial product) per split, splits x (m x n), reduced afterwards
};

struct OzItem {
  int job, tm, tn, z, st0, nst;
};

__device__ __forceinline__ OzItem oz_item(const OzJob* jobs, int njobs, int64_t item) {
  int lo = 0, hi = njobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].item_base <= item) lo = mid; else hi = mid - 1;
  }
  const OzJob& jb = jobs[lo];
  const int64_t local = item - jb.item_base;
  const int per = jb.tiles_m * jb.tiles_n;
  OzItem it;
  it.job = lo;
  it.z = (int)(local / per);
  const int t2 = (int)(local % per);
  it.tm = t2 % jb.tiles_m;
  it.tn = t2 / jb.tiles_m;
  it.st0 = it.z * jb.kst;
  it.nst = min(jb.nst - it.st0, jb.kst);
  return it;
}

// Persistent: CTA b takes items b, b + gridDim.x, ...; tensor memory, the mbarriers and the
// shared-memory ring stay with the CTA across items, and every role counts stages and periods on
// through them, so each barrier's phases are known.  A wait that gives up sets s_gave_up, which
// every other wait sees; all roles then leave their loops.
__global__ void __launch_bounds__(OZ_NT, 1) k_oz_mma(const OzJob* jobs, int njobs, int64_t nitems, int* status) {
  extern __shared__ __align__(1024) unsigned char oz_smem[];
  __shared__ uint32_t s_tmem;
  __shared__ __align__(8) uint64_t s_empty[OZ_RING];  // MMAs of the buffer's stage done
  __shared__ __align__(8) uint64_t s_full[OZ_RING];   // the buffer's stage has landed
  __shared__ __align__(8) uint64_t s_acc[2];          // period's MMAs done; accumulators read
  __shared__ int s_gave_up;
  __shared__ OzItem s_next[OZ_EPI / 32];              // each output warp's next item
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&s_tmem)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int b = 0; b < OZ_RING; ++b) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_empty[b])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_full[b])));
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_acc[0])));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 16;" ::"r"(smem_u32(&s_acc[1])));
    s_gave_up = 0;
  }
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = s_tmem;
  const uint32_t ring = smem_u32(oz_smem);
  constexpr int per_flush = OZ_FLUSH / OZ_BK;

  if (warp == OZ_EPI / 32) {
    // ---- copies
    if (lane == 0) {
      uint32_t G = 0;
      bool ok = true;
      OzItem nx = oz_item(jobs, njobs, blockIdx.x);
      for (int64_t item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
        const OzItem it = nx;
        if (item + gridDim.x < nitems) nx = oz_item(jobs, njobs, item + gridDim.x);
        const OzJob& jb = jobs[it.job];
        const int planes = jb.nim > 0 ? OZ_NSUB : jb.nre;
        const uint32_t ab = 2u * (uint32_t)planes * OZ_A_PL;
        const unsigned char* a = reinterpret_cast<const unsigned char*>(jb.Ad) + ((int64_t)it.tm * jb.nst + it.st0) * ab;
        const unsigned char* b = reinterpret_cast<const unsigned char*>(jb.Bd) + ((int64_t)it.tn * jb.nst + it.st0) * OZ_B_ST;
        for (int st = 0; st < it.nst; ++st, ++G) {
          const int buf = (int)(G % OZ_RING);
          if (G >= OZ_RING && !oz_wait(smem_u32(&s_empty[buf]), (G / OZ_RING - 1) & 1u, &s_gave_up)) {
            ok = false;
            break;
          }
          const uint32_t dst = ring + buf * OZ_STAGE, bar = smem_u32(&s_full[buf]);
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(ab + OZ_B_ST)
                       : "memory");
          oz_copy(dst, a + (int64_t)st * ab, ab, bar);
          oz_copy(dst + OZ_A_ST, b + (int64_t)st * OZ_B_ST, OZ_B_ST, bar);
        }
      }
    }
  } else if (warp == OZ_EPI / 32 + 1) {
    // ---- MMAs
    if (lane == 0) {
      uint32_t G = 0, P = 0;
      bool ok = true;
      OzItem nx = oz_item(jobs, njobs, blockIdx.x);
      for (int64_t item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
        const OzItem it = nx;
        if (item + gridDim.x < nitems) nx = oz_item(jobs, njobs, item + gridDim.x);
        const int nre = jobs[it.job].nre, nim = jobs[it.job].nim;
        const uint32_t lbo_a = (uint32_t)(nim > 0 ? OZ_NSUB : nre) * OZ_A_PL;
        for (int st = 0; st < it.nst; ++st, ++G) {
          const bool fresh = st % per_flush == 0;
          // the last period's accumulators have been read
          if (fresh && P > 0 && !oz_wait(smem_u32(&s_acc[1]), (P - 1) & 1u, &s_gave_up)) {
            ok = false;
            break;
          }
          const int buf = (int)(G % OZ_RING);
          if (!oz_wait(smem_u32(&s_full[buf]), (G / OZ_RING) & 1u, &s_gave_up)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t sa = ring + buf * OZ_STAGE, sb = sa + OZ_A_ST;
          const uint64_t dA = oz_desc(sa, lbo_a), dB = oz_desc(sb, OZ_NSUB * OZ_B_PL);
          // digit i of A against digits 0..6-i of B in one MMA: B's digit planes lie one after
          // another (32 rows each), and level l = i + j sits in columns 32 l (re) and
          // 256 + 32 l (im), so the product lands in the levels i..6 at once.  Digits of A known to
          // be zero (nre, nim) are skipped; digit 0 of the real part always runs, as it opens
          // each period's accumulators.
#pragma unroll
          for (int i = 0; i < OZ_S; ++i) {
            const int N = OZ_BN * (OZ_S - i);
            const uint32_t ip = oz_idesc(false, N), in = oz_idesc(true, N);
            const uint64_t ar = dA + (uint64_t)(i * (OZ_A_PL >> 4)), ai = dA + (uint64_t)((OZ_S + i) * (OZ_A_PL >> 4));
            const uint64_t br = dB, bi = dB + (uint64_t)(OZ_S * (OZ_B_PL >> 4));
            const uint32_t dre = tmem + OZ_BN * i, dim = tmem + 256 + OZ_BN * i;
            const uint32_t first = (fresh && i == 0) ? 0u : 1u;
            if (i < nre) {
              oz_mma(dre, ar, br, ip, first);  // re += Ar Br
              oz_mma(dim, ar, bi, ip, first);  // im += Ar Bi
            }
            if (i < nim) {
              oz_mma(dre, ai, bi, in, 1u);  // re -= Ai Bi
              oz_mma(dim, ai, br, ip, 1u);  // im += Ai Br
            }
          }
          oz_commit(smem_u32(&s_empty[buf]));
          if (st % per_flush == per_flush - 1 || st == it.nst - 1) {
            oz_commit(smem_u32(&s_acc[0]));
            ++P;
          }
        }
      }
    }
  } else {
    // ---- accumulators and outputs: row 32 (warp mod 4) + lane, columns 8 (warp / 4) ..
    const uint32_t base = tmem + ((uint32_t)((warp & 3) * 32) << 16) + OZ_EC * (warp >> 2);
    uint32_t P = 0;
    bool ok = true;
    if (lane == 0) s_next[warp] = oz_item(jobs, njobs, blockIdx.x);
    __syncwarp();
    for (int64_t item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
      // what the outputs need is fetched before the wait for the accumulators, the next item too
      const OzItem it = s_next[warp];
      __syncwarp();
      if (lane == 0 && item + gridDim.x < nitems) s_next[warp] = oz_item(jobs, njobs, item + gridDim.x);
      const OzJob& jb = jobs[it.job];
      const int row = it.tm * OZ_BM + (warp & 3) * 32 + lane, c0 = it.tn * OZ_BN + OZ_EC * (warp >> 2);
      const int er = row < jb.m ? jb.Er[row] : 0;
      const int ecl = c0 + (lane & 7) < jb.n ? jb.Ec[c0 + (lane & 7)] : 0;  // column c's in lane c
      const bool with_beta = jb.splits == 1 && (jb.beta.x != 0.0 || jb.beta.y != 0.0);
      const int64_t step = jb.splits > 1 ? jb.m : jb.transC ? 1 : jb.ldc;
      cplx* out = jb.splits > 1 ? jb.W + ((int64_t)it.z * jb.n + c0) * jb.m + row
                  : jb.transC   ? jb.C + (int64_t)row * jb.ldc + c0
                                : jb.C + (int64_t)c0 * jb.ldc + row;
      const int nc = row < jb.m ? min(OZ_EC, jb.n - c0) : 0;
      long long Rh[2][OZ_EC], Rl[2][OZ_EC];  // sums of levels 0..3 in units of level 3, and 4..6 of level 6
#pragma unroll
      for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int c = 0; c < OZ_EC; ++c) Rh[p][c] = Rl[p][c] = 0;
      const int periods = (it.nst + per_flush - 1) / per_flush;
      for (int q = 0; q < periods; ++q, ++P) {
        if (!oz_wait(smem_u32(&s_acc[0]), P & 1u, &s_gave_up)) ok = false;
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
        for (int p = 0; p < 2; ++p) {
          uint32_t a[OZ_EC], b[OZ_EC] = {};
#pragma unroll
          for (int l = 0; l < OZ_S; l += 2) {
            tmem_ld8(base + 256 * p + OZ_BN * l, a);
            if (l + 1 < OZ_S) tmem_ld8(base + 256 * p + OZ_BN * (l + 1), b);
            tmem_wait(a, b);
#pragma unroll
            for (int c = 0; c < OZ_EC; ++c) {
              const long long x = __float2int_rn(__uint_as_float(a[c]));
              if (l < 4) Rh[p][c] += x * (1 << (7 * (3 - l)));
              else Rl[p][c] += x * (1 << (7 * (6 - l)));
              if (l + 1 < OZ_S) {
                const long long y = __float2int_rn(__uint_as_float(b[c]));
                if (l + 1 < 4) Rh[p][c] += y * (1 << (7 * (2 - l)));
                else Rl[p][c] += y * (1 << (7 * (5 - l)));
              }
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0)
          asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&s_acc[1])) : "memory");
      }
      if (!ok) break;
      const cplx al = jb.alpha, be = jb.beta;
      const bool unit = al.x == 1.0 && al.y == 0.0, minus = al.x == -1.0 && al.y == 0.0;
      const bool unit_beta = be.x == 1.0 && be.y == 0.0;
      // how wide the sums are: |hi| < 2^41 for every value of the warp, or < 2^51, or more
      long long ah = 0;
#pragma unroll
      for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int c = 0; c < OZ_EC; ++c) ah |= Rh[p][c] ^ (Rh[p][c] >> 63);
      const int width = __all_sync(0xffffffffu, ah < (1ll << 41)) ? 0 : __all_sync(0xffffffffu, ah < (1ll << 51)) ? 1 : 2;
#pragma unroll
      for (int cb = 0; cb < OZ_EC; cb += 4) {
        cplx old[4];  // four loads in flight: a store to C orders the loads after it
        if (with_beta) {
#pragma unroll
          for (int c = 0; c < 4; ++c)
            if (cb + c < nc) old[c] = out[(cb + c) * step];
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int ec = __shfl_sync(0xffffffffu, ecl, cb + c);
          if (cb + c >= nc) continue;
          const int sc = er + ec - 56;  // 14 and the six digits below level 0
          cplx v = cmk(oz_value(Rh[0][cb + c], Rl[0][cb + c], sc, width), oz_value(Rh[1][cb + c], Rl[1][cb + c], sc, width));
          if (minus) v = cmk(-v.x, -v.y);
          else if (!unit) v = cmk(al.x * v.x - al.y * v.y, al.x * v.y + al.y * v.x);
          if (with_beta) v = unit_beta ? cadd(old[c], v) : cfma(be, old[c], v);
          out[(cb + c) * step] = v;
        }
      }
      __syncwarp();  // the accumulator reads are warp-wide
    }
  }
  __syncwarp();
  __syncthreads();
  if (s_gave_up && tid == 0) {
    // a wait gave up: let the copies and MMAs in flight drain (bounded) before freeing
    // tensor memory and leaving the shared memory they write
    for (int b = 0; b < OZ_RING; ++b)
      for (uint32_t par = 0; par < 2; ++par) {
        int mine = 0;
        oz_wait(smem_u32(&s_full[b]), par, &mine);
        mine = 0;
        oz_wait(smem_u32(&s_empty[b]), par, &mine);
      }
    atomicExch(status, 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
}

// C = beta C + sum_s W_s (fixed order).
__global__ void k_oz_reduce(const cplx* W, int m, int n, int splits, cplx beta, cplx* C, int ldc, int transC) {
  const int64_t tot = (int64_t)m * n;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e % m);
    const int64_t j = e / m;
    cplx acc = cmk(0.0, 0.0);
    for (int s = 0; s < splits; ++s) acc = cadd(acc, W[s * tot + e]);
    cplx* c = transC ? C + (int64_t)i * ldc + j : C + j * ldc + i;
    if (beta.x != 0.0 || beta.y != 0.0) acc = cfma(beta, *c, acc);
    *c = acc;
  }
}

}  // namespace

// Products worth the tensor cores: k >= 96 and half a tile's rows.  (At most 2^26 values of k: the 64-bit sums hold
// 2^27.)  Shorter ones stay in double-float although they were faster here (690 x 2048 x 49 0.112 ms against
// 0.165): the digit planes' error is relative to the largest entry of a row and a column, double-float's to each
// term.  Against FP64 on the operands of the builds the short products' normwise error was up to 24 times
// double-float's (8.9e-13 and 3.7e-14 for 138 x 72 x 72), and operands graded over 12 decades left 4e-4 for 2e-14.
bool ozaki_eligible(const GemmJob& j) { return j.k >= 96 && j.k <= (1 << 26) && j.m >= 48 && j.n >= 8; }

// A batch of products on the tensor cores (see the head of this file): exponents and digit
// planes of every operand (two launches), one persistent MMA launch over all tiles, and a
// fixed-order reduction for the products split along k.
void ozaki_gemm_batched(const std::vector<GemmJob>& js, cudaStream_t s) {
  if (js.empty()) return;
  static const int sms = [] {
    int dev = 0, sm = 0;
    HBS_CUDA(cudaGetDevice(&dev));
    HBS_CUDA(cudaDeviceGetAttribute(&sm, cudaDevAttrMultiProcessorCount, dev));
    return sm;
  }();
  static const bool attr = [] {
    HBS_CUDA(cudaFuncSetAttribute(k_oz_mma, cudaFuncAttributeMaxDynamicSharedMemorySize, OZ_SMEM));
    return true;
  }();
  (void)attr;
  const int nj = (int)js.size();
  std::vector<OzJob> oj(nj);
  int64_t adig = 0, bdig = 0, eA = 0, eB = 0, wtot = 0, items = 0;
  double tflops = 0.0;
  int tiles_all = 0;
  for (int q = 0; q < nj; ++q) {
    const GemmJob& j = js[q];
    OzJob& o = oj[q];
    o.m = j.m;
    o.n = j.n;
    o.tiles_m = (j.m + OZ_BM - 1) / OZ_BM;
    o.tiles_n = (j.n + OZ_BN - 1) / OZ_BN;
    o.nst = (j.k + OZ_BK - 1) / OZ_BK;  // stages of 16; the last period may be short
    o.nre = j.a_real_digits > 0 ? std::min(j.a_real_digits, OZ_S) : OZ_S;
    o.nim = j.a_real_digits > 0 ? 0 : OZ_S;
    tiles_all += o.tiles_m * o.tiles_n;
  }
  for (int q = 0; q < nj; ++q) {
    const GemmJob& j = js[q];
    OzJob& o = oj[q];
    // split along k (in whole periods) only when the whole batch has too few tiles to fill the SMs
    constexpr int kPer = OZ_FLUSH / OZ_BK;
    const int periods = (o.nst + kPer - 1) / kPer;
    o.splits = 1;
    if (tiles_all < sms && j.k >= 4096) o.splits = std::max(1, std::min(periods, sms / std::max(1, tiles_all)));
    o.kst = (periods + o.splits - 1) / o.splits * kPer;
    o.splits = (o.nst + o.kst - 1) / o.kst;
    o.item_base = items;
    items += (int64_t)o.tiles_m * o.tiles_n * o.splits;
    o.alpha = j.alpha;
    o.beta = j.beta;
    o.C = j.C;
    o.ldc = j.ldc;
    o.transC = j.transC;
    o.Ad = reinterpret_cast<const unsigned short*>(adig);  // offsets for now
    o.Bd = reinterpret_cast<const unsigned short*>(bdig);
    o.Er = reinterpret_cast<const int*>(eA);
    o.Ec = reinterpret_cast<const int*>(eB);
    o.W = reinterpret_cast<cplx*>(o.splits > 1 ? wtot : 0);
    const int64_t mpad = (int64_t)o.tiles_m * OZ_BM, npad = (int64_t)o.tiles_n * OZ_BN, Kpad = (int64_t)o.nst * OZ_BK;
    adig += (o.nim > 0 ? OZ_NSUB : o.nre) * mpad * Kpad;
    bdig += OZ_NSUB * npad * Kpad;
    eA += j.m;
    eB += j.n;
    if (o.splits > 1) wtot += (int64_t)o.splits * j.m * j.n;
    // executed: per digit i of A, 2 (7 - i) MMA units for its real part, 2 (7 - i) for its
    // imaginary part; 112 units in all for a general A (224 flops per m n k)
    double units = 0.0;
    for (int i = 0; i < OZ_S; ++i) units += 2.0 * (OZ_S - i) * ((i < o.nre) + (i < o.nim));
    tflops += 2.0 * units * mpad * (double)npad * Kpad;
  }
  DevBuf<unsigned short> Ad(adig), Bd(bdig);
  DevBuf<int> E(eA + eB), st(1);
  DevBuf<cplx> W(std::max<int64_t>(wtot, 1));
  std::vector<OzOperand> ops;
  ops.reserve(2 * nj);
  int64_t maxexp = 1, maxdig = 1;
  for (int q = 0; q < nj; ++q) {
    const GemmJob& j = js[q];
    OzJob& o = oj[q];
    unsigned short* ad = Ad.get() + reinterpret_cast<int64_t>(o.Ad);
    unsigned short* bd = Bd.get() + reinterpret_cast<int64_t>(o.Bd);
    int* er = E.get() + reinterpret_cast<int64_t>(o.Er);
    int* ec = E.get() + eA + reinterpret_cast<int64_t>(o.Ec);
    // op(A) row r, k: transA ? A[r lda + k] : A[k lda + r];  B^T row c, k: B[c ldb + k]
    const int mpad = o.tiles_m * OZ_BM, npad = o.tiles_n * OZ_BN, Kpad = o.nst * OZ_BK;
    ops.push_back({j.A, j.lda, j.transA ? 1 : 0, j.m, j.k, mpad, Kpad, OZ_BM, o.nim > 0 ? OZ_NSUB : o.nre, er, ad});
    ops.push_back({j.B, j.ldb, 1, j.n, j.k, npad, Kpad, OZ_BN, OZ_NSUB, ec, bd});
    o.Ad = ad;
    o.Bd = bd;
    o.Er = er;
    o.Ec = ec;
    o.W = o.splits > 1 ? W.get() + reinterpret_cast<int64_t>(o.W) : nullptr;
    maxexp = std::max(maxexp, (int64_t)((std::max(j.m, j.n) + 31) / 32) * ((j.k + 1023) / 1024));
    maxdig = std::max(maxdig, (int64_t)std::max(mpad, npad) * (Kpad / 8));
  }
  HBS_CUDA(cudaMemsetAsync(st.get(), 0, sizeof(int), s));
  HBS_CUDA(cudaMemsetAsync(E.get(), 0x80, sizeof(int) * (size_t)(eA + eB), s));  // below every exponent
  DevBuf<OzOperand> dops(ops.size());
  HBS_CUDA(cudaMemcpyAsync(dops.get(), ops.data(), ops.size() * sizeof(OzOperand), cudaMemcpyHostToDevice, s));
  {
    prof::KScope _ks("k_oz_digits", s);
    const unsigned bx_e = (unsigned)std::min<int64_t>(4096, maxexp);
    const unsigned bx_d = (unsigned)std::min<int64_t>(8192, (maxdig + 255) / 256);
    for (size_t o0 = 0; o0 < ops.size(); o0 += 65535) {
      const unsigned ny = (unsigned)std::min<size_t>(65535, ops.size() - o0);
      k_oz_exponents<<<dim3(bx_e, ny), 256, 0, s>>>(dops.get() + o0);
      k_oz_digits<<<dim3(bx_d, ny), 256, 0, s>>>(dops.get() + o0);
    }
  }
  HBS_LAUNCH_CHECK("k_oz_digits");
  DevBuf<OzJob> dj(nj);
  HBS_CUDA(cudaMemcpyAsync(dj.get(), oj.data(), nj * sizeof(OzJob), cudaMemcpyHostToDevice, s));
  {
    // executed tensor work: 28 digit pairs x 4 real products x 2 flops per (padded) m n k
    prof::KScope _ks("k_oz_mma", s, tflops, 0.0);
    const unsigned grid = (unsigned)std::min<int64_t>(sms, items);
    k_oz_mma<<<grid, OZ_NT, OZ_SMEM, s>>>(dj.get(), nj, items, st.get());
  }
  HBS_LAUNCH_CHECK("k_oz_mma");
  for (int q = 0; q < nj; ++q) {
    const OzJob& o = oj[q];
    if (o.splits <= 1) continue;
    prof::KScope _ks("k_oz_reduce", s);
    k_oz_reduce<<<grid_1d((int64_t)o.m * o.n), 256, 0, s>>>(o.W, o.m, o.n, o.splits, o.beta, o.C, o.ldc, o.transC);
  }
  HBS_LAUNCH_CHECK("k_oz_reduce");
  int hs = 0;
  read_to_host(&hs, st.get(), sizeof(int), s);
  if (hs) throw Error(HBS_ERR_TIMEOUT, "tensor-core GEMM: an MMA completion wait gave up");
}

}  // namespace hbs
