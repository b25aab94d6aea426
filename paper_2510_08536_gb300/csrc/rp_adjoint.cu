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
// matrix it was 16 bytes of map an entry and scattered writes.) Cells, faces and
// interface entries are one range, so that a small call is one trip of the grid;
// 32 registers, so that all eight blocks an SM run at once (40: 66 us at 128^3).
// Row by row, then this, us: 16^3 on 8 ranks 2.9, 2.3; 48^3 on 27 4.6, 5.1; 64^3 on 64
// 8.1, 7.3; 128^3 on 8 62.9, 41.5, on 64 60.8, 43.8, on 512 59.3, 46.2; 192^3 on 64 244,
// 154; rows of 15 entries, 1M 149, 43. At 128^3 its FP64 products (64 to 76 clocks a
// warp's) take 55% of the pipe. STREAM: results of more than 2M elements leave L2
// (128^3 on 64 ranks 47.3 us without it, 192^3 151; 64^3 7.3 us, with it 8.4).
// Symmetric storage: one slot holds both coefficients of a face, both gradients are added.
struct GradArgs {
  int32_t k, trips;
  int64_t n, n_faces, n_iface;
  const int64_t *row_off, *slot_off, *face_off, *iface_off;
  const int32_t *lower, *upper, *iface_row, *iface_gcol;
};
template <bool STREAM>
__device__ __forceinline__ void put(double* p, double v) {
  if (STREAM) __stcs(p, v);
  else *p = v;
}
template <bool SHARED_SLOTS, bool STREAM>
__global__ void __launch_bounds__(kThreads, kBlocksPerSm)
    k_entry_grad(const GradArgs a, const double* __restrict__ lam, const double* __restrict__ x,
                 double* __restrict__ g) {
  Walk w = grid_walk(a.trips);
  const double *lr = lam, *xr = x;
  double* out = g;
  int64_t gap = 0;
  for_ranked(
      w, 0, a.n, a.row_off, a.k,
      [&](int r) { out = g + (__ldg(a.slot_off + r) - __ldg(a.row_off + r)); },
      [&](int64_t i) { put<STREAM>(out + i, -__ldg(lam + i) * __ldg(x + i)); });
  for_ranked(
      w, a.n, a.n_faces, a.face_off, a.k,
      [&](int r) {
        const int64_t r0 = __ldg(a.row_off + r), f0 = __ldg(a.face_off + r);
        lr = lam + r0;
        xr = x + r0;
        out = g + (__ldg(a.slot_off + r) + (__ldg(a.row_off + r + 1) - r0) - f0);
        gap = __ldg(a.face_off + r + 1) - f0;
      },
      [&](int64_t f) {
        const int l = STREAM ? __ldcs(a.lower + f) : __ldg(a.lower + f), u = STREAM ? __ldcs(a.upper + f) : __ldg(a.upper + f);
        if (!RP_IN((lr - lam) + l, 0, a.n, kChkGather) || !RP_IN((lr - lam) + u, 0, a.n, kChkGather)) return;
        const double gu = __dmul_rn(-__ldg(lr + l), __ldg(xr + u)), gl = __dmul_rn(-__ldg(lr + u), __ldg(xr + l));
        if (SHARED_SLOTS) {
          put<STREAM>(out + f, __dadd_rn(gu, gl));
        } else {
          put<STREAM>(out + f, gu);
          put<STREAM>(out + f + gap, gl);
        }
      });
  for_ranked(
      w, a.n + a.n_faces, a.n_iface, a.iface_off, a.k,
      [&](int r) {
        const int64_t r0 = __ldg(a.row_off + r), nf = __ldg(a.face_off + r + 1) - __ldg(a.face_off + r);
        lr = lam + r0;
        out = g + (__ldg(a.slot_off + r) + (__ldg(a.row_off + r + 1) - r0) + (SHARED_SLOTS ? 1 : 2) * nf -
                   __ldg(a.iface_off + r));
      },
      [&](int64_t e) {
        const int i = __ldg(a.iface_row + e), j = __ldg(a.iface_gcol + e);
        if (!RP_IN((lr - lam) + i, 0, a.n, kChkGather) || !RP_IN(j, 0, a.n, kChkGather)) return;
        out[e] = -__ldg(lr + i) * __ldg(x + j);
      });
}

// -(lambda_l - lambda_u)(x_l - x_u) per face, then per interface entry, rank by rank
__global__ void __launch_bounds__(kThreads)
    k_face_grad(int k, int64_t total, const int64_t* __restrict__ out_off, const int64_t* __restrict__ row_off,
                const int64_t* __restrict__ face_off, const int64_t* __restrict__ iface_off,
                const int32_t* __restrict__ lower, const int32_t* __restrict__ upper,
                const int32_t* __restrict__ iface_row, const int32_t* __restrict__ iface_gcol,
                const double* __restrict__ lam, const double* __restrict__ x, double* __restrict__ g) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    int r = find_rank(out_off, k, t);
    int64_t u = t - out_off[r];
    int64_t F = face_off[r + 1] - face_off[r];
    int64_t a, b;
    if (u < F) {
      a = row_off[r] + lower[face_off[r] + u];
      b = row_off[r] + upper[face_off[r] + u];
    } else {
      int64_t e = iface_off[r] + (u - F);
      a = row_off[r] + iface_row[e];
      b = iface_gcol[e];
    }
    if (!RP_IN(a, 0, row_off[k], kChkGather) || !RP_IN(b, 0, row_off[k], kChkGather)) continue;
    g[t] = -(lam[a] - lam[b]) * (x[a] - x[b]);
  }
}

// The same through the faces and then the interface entries in runs of eight trips,
// where a search of a rank a run pays: more than 128 ranks. Element by element, then in
// runs, us: 64^3 on 64 ranks 8.9, 11.5; 128^3 on 8 44.2, 44.3, on 64 48.4, 47.4, on 512
// 62.1, 50.5; 192^3 on 64 146.8, 150.6; 4M rows of 15 entries on one 183, 213.
__global__ void __launch_bounds__(kThreads, kBlocksPerSm)
    k_face_grad_runs(const GradArgs a, const double* __restrict__ lam, const double* __restrict__ x,
                     double* __restrict__ g) {
  Walk w = grid_walk(8);
  const double *lr = lam, *xr = x;
  double* out = g;
  // rank r's faces are written after the faces and interface entries of the ranks before it
  for_ranked(
      w, 0, a.n_faces, a.face_off, a.k,
      [&](int r) {
        const int64_t r0 = __ldg(a.row_off + r);
        lr = lam + r0;
        xr = x + r0;
        out = g + __ldg(a.iface_off + r);
      },
      [&](int64_t f) {
        const int l = __ldg(a.lower + f), u = __ldg(a.upper + f);
        if (!RP_IN((lr - lam) + l, 0, a.n, kChkGather) || !RP_IN((lr - lam) + u, 0, a.n, kChkGather)) return;
        out[f] = -(__ldg(lr + l) - __ldg(lr + u)) * (__ldg(xr + l) - __ldg(xr + u));
      });
  for_ranked(
      w, a.n_faces, a.n_iface, a.iface_off, a.k,
      [&](int r) {
        const int64_t r0 = __ldg(a.row_off + r);
        lr = lam + r0;
        xr = x + r0;
        out = g + __ldg(a.face_off + r + 1);
      },
      [&](int64_t e) {
        const int i = __ldg(a.iface_row + e), j = __ldg(a.iface_gcol + e);
        if (!RP_IN((lr - lam) + i, 0, a.n, kChkGather) || !RP_IN(j, 0, a.n, kChkGather)) return;
        out[e] = -(__ldg(lr + i) - __ldg(lam + j)) * (__ldg(xr + i) - __ldg(x + j));
      });
}

inline GradArgs grad_args(const rp_handle* h) {
  return GradArgs{h->k, walk_trips(h, h->n + h->n_face_out), h->n, h->face_off[h->k], h->iface_off[h->k],
                  h->d_row_off, h->d_slot_off, h->d_face_off, h->d_iface_off,
                  h->d_lower, h->d_upper, h->d_iface_row, h->d_iface_gcol};
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
  const int64_t total = h->n + h->n_face_out;
  const int g = grid_for(h, total);
  const bool stream_out = total > 2'000'000;
  const GradArgs a = grad_args(h);
  if (h->symmetric && stream_out) k_entry_grad<true, true><<<g, kThreads, 0, s>>>(a, lambda, x, g_buffer);
  else if (h->symmetric) k_entry_grad<true, false><<<g, kThreads, 0, s>>>(a, lambda, x, g_buffer);
  else if (stream_out) k_entry_grad<false, true><<<g, kThreads, 0, s>>>(a, lambda, x, g_buffer);
  else k_entry_grad<false, false><<<g, kThreads, 0, s>>>(a, lambda, x, g_buffer);
  RP_TRY_CUDA(cudaGetLastError());
  return RP_OK;
}

extern "C" rp_status rp_face_grad(rp_handle* h, const double* lambda, const double* x, double* g_face,
                                  void* stream) {
  if (!h || (!lambda && h->n) || (!x && h->n) || (!g_face && h->n_face_out)) return fail(RP_EINVAL, "null argument");
  if (h->n_face_out == 0) return RP_OK;
  cudaStream_t s = (cudaStream_t)stream;
  const int g = grid_for(h, h->n_face_out);
  if (h->k > 128)
    k_face_grad_runs<<<g, kThreads, 0, s>>>(grad_args(h), lambda, x, g_face);
  else
    k_face_grad<<<g, kThreads, 0, s>>>(h->k, h->n_face_out, h->d_out_off, h->d_row_off, h->d_face_off, h->d_iface_off,
                                       h->d_lower, h->d_upper, h->d_iface_row, h->d_iface_gcol, lambda, x, g_face);
  RP_TRY_CUDA(cudaGetLastError());
  return RP_OK;
}
