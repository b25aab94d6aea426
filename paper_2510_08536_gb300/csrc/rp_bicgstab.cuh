// Arguments of BiCGStab, shared by its two forms: the streaming kernels B1-B5
// (rp_bicgstab.cu) and the resident kernel (rp_resident_bs.cu).
#pragma once

#include "rp_common.cuh"
#include "rp_resident.cuh"

namespace rp {

struct BsCtl {
  double bb, thresh, tol, rr, ss;
  double rho, rho_old, alpha, omega;
  double ithresh, inner_tol;  // the inner loop's target: thresh (FP64); inner_tol^2 (r32, r32) (mixed)
  int32_t iter, max_iter, stop, status, pass, restarts, max_restarts, half, x_zero;
  int32_t outer, max_outer;
  unsigned int ticket;
};

// the vectors and the matrix of one working precision
template <typename T>
struct BsVecs {
  const T* vals;
  const T* dinv;
  Parts<T> parts;
  Sliced<T> sl;
  T *r, *rhat, *p, *v, *s, *t, *phat, *shat;
  T* x;  // FP32: the correction d; FP64: unused (the caller's x, through SolveIO)
};

struct BsArgs {
  int64_t n;
  const int32_t* row_ptr;
  const int32_t* col;
  BsVecs<double> d;  // FP64 solve; its matrix also serves the residual passes
  BsVecs<float> f;   // FP32 inner solve (mixed)
  BsCtl* c;
  SolveIO* io;
  double* partials;
  cudaGraphConditionalHandle inner, outer;
  int in_graph;
};

// The resident form of the inner loop: one cooperative launch runs every
// iteration (cap: at most that many, then the state is left in memory for the
// next launch).
template <typename T>
struct ResidentBsArgs {
  BsArgs a;
  unsigned int* sync;  // memory of the grid barrier and sums, cleared before each solve
  int64_t spin;        // probe limit of a barrier wait
  int32_t rows;        // rows of shared memory a block holds (a multiple of 32)
  int32_t cap;
};
// Its launch, or fn = nullptr where four vectors do not fit the chip's shared memory.
template <typename T>
ResidentPlan resident_bs_plan(const rp_handle* h, const BsVecs<T>& v);

}  // namespace rp
