// Host interface of the blocked Gauss-Jordan elimination (gjx.cu).
#pragma once

#include <string>
#include <vector>

#include "common.cuh"
#include "devbuf.hpp"

namespace hbs {

// One system: A (n x n, ld n) and q right-hand sides B (n x q, ld n), complex128 on the device.
struct GjxSys {
  cplx* A;
  cplx* B;
  int n, q;
};

// The same on the device, with the working copies that the elimination runs on (complex128 or
// double-float pairs) and its records.
struct GjxMat {
  void* A;
  void* B;
  cplx* srcA;
  cplx* srcB;
  int n, q;
  int* piv;      // n: pivot row of each column
  int* colof;    // n: column a row was pivot of, -1 before
  double* pmag;  // n: squared modulus of each pivot
  int* singular;
};

// An elimination's state: the exchanged matrices stay in A for gjx_solution and gjx_apply.
struct Gjx {
  int nm = 0, nmax = 0, qmax = 0;
  bool df = false;
  DevBuf<GjxMat> mats;
  DevBuf<cplx> A, B;
  DevBuf<int> piv, colof, sing;
  DevBuf<double> pmag;
};

// Whether clusters of cs CTAs hold panels of nmax rows, the default cluster size, and the tuned one.
bool gjx_cluster_fits(int cs, int nmax);
int gjx_cluster(int nm, int nmax, bool df);
int gjx_tuned_cluster(const std::string& tkey, int nm, int nmax, bool df);

// Eliminates every system (invert: all columns; else the columns to the right and the
// right-hand sides only).  An FP64 solve eliminates in A itself, everything else in a copy; B is
// only read.
void gjx_eliminate(Gjx& g, const std::vector<GjxSys>& sys, bool df, bool invert, int cs, cudaStream_t s);
// After a solve: out[m] (n x q) = the solutions, illcond[m] = 1 if a pivot is 1e-14 of the largest, zero or not finite.
void gjx_solution(Gjx& g, cplx* const* out, int* illcond, cudaStream_t s);
// After a double-float solve: out[m] += the elimination applied to res[m] (n x q each) in FP64 arithmetic.  Once:
// the eliminated matrices are FP64 afterwards.
void gjx_apply(Gjx& g, const cplx* const* res, cplx* const* out, cudaStream_t s);
// In-place inverses; throws HBS_WARN_ILLCOND on a block that is singular or not finite.
void gjx_invert(const std::vector<std::pair<cplx*, int>>& mats, cudaStream_t s, const char* what);

}  // namespace hbs
