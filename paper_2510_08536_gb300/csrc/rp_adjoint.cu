// Adjoint solve and gradients of the merged system.
//
// With A x = b and a loss L(x), the adjoint lambda solves A^T lambda = dL/dx;
// then dL/db = lambda and dL/da_ij = -lambda_i x_j for every stored entry.
// A^T reuses A's pattern: valsT[p] = vals[tpos[p]] (one gather pass), and the
// Jacobi diagonal is unchanged by transposition; the sliced layout of A then
// serves A^T with its values gathered from valsT. Symmetric storage needs no
// transpose at all.
#include <algorithm>

#include "rp_common.cuh"

namespace rp {

rp_status solve_common(rp_handle* h, int mode, const double* vals, const double* dinv, SolveGraph* slot,
                        const double* b, double* x, double tol, int32_t x_is_guess, int32_t where,
                        rp_solve_info* info, cudaStream_t s);

__global__ void __launch_bounds__(kThreads)
    k_transpose_vals(int64_t nnz, const int32_t* __restrict__ tpos, const double* __restrict__ vals,
                     double* __restrict__ valsT) {
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nnz; p += (int64_t)gridDim.x * blockDim.x) {
    const int32_t t = __ldg(tpos + p);
    valsT[p] = RP_IN(t, 0, nnz, kChkTranspose) ? __ldg(vals + t) : 0.0;
  }
}

// dL/da_ij = -lambda_i x_j for every slot of the buffer, in the buffer's own
// order: the diagonal, upper, lower and interface coefficients of each rank are
// runs of the addressing the handle keeps, so a face's two rows are read once for
// both of its slots and every write is coalesced. (Row by row over the merged
// matrix it was 16 bytes of map an entry and scattered writes.) At 128^3 48 us, its
// FP64 products (64 to 76 clocks a warp's) 55% of the pipe; 32 registers, so that all
// eight blocks an SM run at once (40: 66 us). With the faces 112.8 -> 105.2 us. Symmetric
// storage: one slot holds both coefficients of a face, both gradients are added.
struct GradArgs {
  int32_t k;
  const int64_t *row_off, *slot_off, *face_off, *iface_off;
  const int32_t *lower, *upper, *iface_row, *iface_gcol;
};
template <bool SHARED_SLOTS>
__global__ void __launch_bounds__(kThreads, kBlocksPerSm)
    k_entry_grad(const GradArgs a, const double* __restrict__ lam, const double* __restrict__ x,
                 double* __restrict__ g) {
  const int64_t n = __ldg(a.row_off + a.k);
  for_ranked(a.row_off, a.k, [&](int r, int64_t i) {
    __stcs(g + __ldg(a.slot_off + r) + (i - __ldg(a.row_off + r)), -__ldg(lam + i) * __ldg(x + i));
  });
  for_ranked(a.face_off, a.k, [&](int r, int64_t f) {
    const int64_t r0 = __ldg(a.row_off + r), nc = __ldg(a.row_off + r + 1) - r0, f0 = __ldg(a.face_off + r);
    const int64_t l = r0 + __ldcs(a.lower + f), u = r0 + __ldcs(a.upper + f);
    if (!RP_IN(l, 0, n, kChkGather) || !RP_IN(u, 0, n, kChkGather)) return;
    const double gu = __dmul_rn(-__ldg(lam + l), __ldg(x + u)), gl = __dmul_rn(-__ldg(lam + u), __ldg(x + l));
    double* out = g + __ldg(a.slot_off + r) + nc + (f - f0);
    if (SHARED_SLOTS) {
      __stcs(out, __dadd_rn(gu, gl));
    } else {
      __stcs(out, gu);
      __stcs(out + (__ldg(a.face_off + r + 1) - f0), gl);
    }
  });
  for_ranked(a.iface_off, a.k, [&](int r, int64_t e) {
    const int64_t r0 = __ldg(a.row_off + r), nc = __ldg(a.row_off + r + 1) - r0;
    const int64_t nf = __ldg(a.face_off + r + 1) - __ldg(a.face_off + r);
    const int64_t i = r0 + a.iface_row[e], j = a.iface_gcol[e];
    if (!RP_IN(i, 0, n, kChkGather) || !RP_IN(j, 0, n, kChkGather)) return;
    g[__ldg(a.slot_off + r) + nc + (SHARED_SLOTS ? 1 : 2) * nf + (e - __ldg(a.iface_off + r))] =
        -__ldg(lam + i) * __ldg(x + j);
  });
}

// -(lambda_l - lambda_u)(x_l - x_u) per face, then per interface entry, rank by rank
__global__ void __launch_bounds__(kThreads)
    k_face_grad(const GradArgs a, const double* __restrict__ lam, const double* __restrict__ x,
                double* __restrict__ g) {
  const int64_t n = __ldg(a.row_off + a.k);
  auto put = [&](int64_t at, int64_t i, int64_t j) {
    if (!RP_IN(i, 0, n, kChkGather) || !RP_IN(j, 0, n, kChkGather)) return;
    __stcs(g + at, -(__ldg(lam + i) - __ldg(lam + j)) * (__ldg(x + i) - __ldg(x + j)));
  };
  // rank r's faces are written after the faces and interface entries of the ranks before it
  for_ranked(a.face_off, a.k, [&](int r, int64_t f) {
    const int64_t r0 = __ldg(a.row_off + r);
    put(f + __ldg(a.iface_off + r), r0 + __ldcs(a.lower + f), r0 + __ldcs(a.upper + f));
  });
  for_ranked(a.iface_off, a.k, [&](int r, int64_t e) {
    put(e + __ldg(a.face_off + r + 1), __ldg(a.row_off + r) + a.iface_row[e], a.iface_gcol[e]);
  });
}

inline GradArgs grad_args(const rp_handle* h) {
  return GradArgs{h->k,       h->d_row_off, h->d_slot_off,  h->d_face_off, h->d_iface_off,
                  h->d_lower, h->d_upper,   h->d_iface_row, h->d_iface_gcol};
}

RP_CHECK_TU(adjoint)

}  // namespace rp

using namespace rp;

extern "C" rp_status rp_solve_adjoint(rp_handle* h, const double* g, double* lambda, double tol,
                                      rp_solve_info* info, void* stream) {
  if (!h || (!g && h->n) || (!lambda && h->n)) return fail(RP_EINVAL, "null argument");
  if (!(tol >= 0.0)) return fail(RP_EINVAL, "tol must be >= 0");
  if (h->n_parts != 1) return fail(RP_EUNSUPPORTED, "adjoint solve needs n_parts == 1");
  if (h->n == 0) {
    if (info) *info = rp_solve_info{RP_OK, 0, 0, 0, 0, 0.0};
    return RP_OK;
  }
  cudaStream_t s = (cudaStream_t)stream;
  if (h->symmetric)
    return solve_common(h, false, h->vals, h->dinv, &h->graphs.fp64, g, lambda, tol, 0, RP_MEM_DEVICE, info, s);
  if (!h->tpos) return fail(RP_EINVAL, "adjoint of general storage needs want_transpose");
  if (!h->valsT) {
    cudaError_t e = cudaMalloc((void**)&h->valsT, sizeof(double) * (h->nnz + 64));
    if (e != cudaSuccess) {
      h->valsT = nullptr;
      cudaGetLastError();
      return fail(RP_ENOMEM, "cudaMalloc of transposed values failed");
    }
  }
  k_transpose_vals<<<grid_for(h, h->nnz), kThreads, 0, s>>>(h->nnz, h->tpos, h->vals, h->valsT);
  RP_TRY_CUDA(cudaGetLastError());
  RP_TRY(fill_sliced_transposed(h, s));  // the iteration multiplies with the sliced layout of A^T
  return solve_common(h, false, h->valsT, h->dinv, &h->graphs.adjoint, g, lambda, tol, 0, RP_MEM_DEVICE, info, s);
}

extern "C" rp_status rp_entry_grad(rp_handle* h, const double* lambda, const double* x, double* g_buffer,
                                   void* stream) {
  if (!h || (!lambda && h->n) || (!x && h->n) || (!g_buffer && h->n_slots)) return fail(RP_EINVAL, "null argument");
  if (h->n_parts != 1) return fail(RP_EUNSUPPORTED, "entry gradients need n_parts == 1");
  if (h->n == 0) return RP_OK;
  cudaStream_t s = (cudaStream_t)stream;
  const int g = grid_for(h, std::max<int64_t>(h->n, h->n_face_out) / 4);
  if (h->symmetric) k_entry_grad<true><<<g, kThreads, 0, s>>>(grad_args(h), lambda, x, g_buffer);
  else k_entry_grad<false><<<g, kThreads, 0, s>>>(grad_args(h), lambda, x, g_buffer);
  RP_TRY_CUDA(cudaGetLastError());
  return RP_OK;
}

extern "C" rp_status rp_face_grad(rp_handle* h, const double* lambda, const double* x, double* g_face,
                                  void* stream) {
  if (!h || (!lambda && h->n) || (!x && h->n) || (!g_face && h->n_face_out)) return fail(RP_EINVAL, "null argument");
  if (h->n_face_out == 0) return RP_OK;
  cudaStream_t s = (cudaStream_t)stream;
  k_face_grad<<<grid_for(h, h->n_face_out / 4), kThreads, 0, s>>>(grad_args(h), lambda, x, g_face);
  RP_TRY_CUDA(cudaGetLastError());
  return RP_OK;
}
