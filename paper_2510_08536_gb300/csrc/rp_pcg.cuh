// Arguments of the PCG iteration, shared by its two forms: the streaming
// kernels K1-K3 (rp_pcg.cu) and the resident kernel (rp_resident.cu).
#pragma once

#include "rp_common.cuh"
#include "rp_resident.cuh"

namespace rp {

template <typename T>
struct IterArgs {
  int64_t n;
  const int32_t* row_ptr;
  const int32_t* col;
  const T* vals;
  const T* dinv;
  T* r;
  T* p;
  T* q;
  T* xd;  // iterate updated by K3: the correction d (mixed); nullptr = io->x
  Ctl* ctl;
  SolveIO* io;
  double* partials;
  cudaGraphConditionalHandle inner;
  int in_graph;  // 0: launched on a stream (kernel timing), no condition to set
  Parts<T> parts;
  Sliced<T> sl;  // K1 runs k_it_spmv_sl when built (n_slices > 0)
  Line<T> line;  // line preconditioner (K2 writes z, K3 reads it); l == nullptr: Jacobi
};

// The resident form of the inner iteration: one cooperative launch runs every
// iteration of an inner run (cap: at most that many, then the state is left in
// memory for the next launch).
template <typename T>
struct ResidentArgs {
  IterArgs<T> it;
  unsigned int* sync;  // memory of the grid barrier and sums, cleared before each solve
  int64_t spin;        // probe limit of a barrier wait
  int32_t rows;        // rows of shared memory a block holds (a multiple of 32)
  int32_t width;       // longest row of a kept matrix
  int32_t cap;
};
// The launch of the resident kernel for these arguments, or fn = nullptr where
// the vectors of the iteration do not fit the chip's shared memory.
template <typename T>
ResidentPlan resident_plan(const rp_handle* h, const IterArgs<T>& a, bool scaled);

}  // namespace rp
