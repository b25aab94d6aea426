// The resident form of the PCG iteration: one cooperative launch (one block an
// SM) runs a whole inner run, with the vectors in shared memory.
//
// The streaming form (K1, K2, K3 of rp_pcg.cu in a conditional graph) costs
// 20 us an iteration however small the system is: three launches, two block
// elections and the latency of cold pipelines. Systems whose vectors fit the
// SMs' shared memory (152 x 227 KB) need none of it: block b owns a contiguous
// run of 32-row slices and keeps r, x, p and q of those rows in shared memory;
// only p, which the products gather across blocks, is also written to global
// memory. The grid meets three times an iteration:
//   A  q = A p,                             (p, q)          | sum -> alpha
//   B  r -= alpha q, z = D^-1 r, x += alpha p, (r, z), (r, r) | sum -> beta, stop test
//   C  p = z + beta p                                       | barrier
// with the arithmetic of K1-K3, row by row the same fused multiply-adds. The sums
// are the same integers in every block (grid_sum_unit), so all blocks hold the same
// scalars and take the same branches.
//
// Forms (resident_plan takes the first that fits; on layouts other than the uniform one
// within the lines at plan_resident):
//   matrix kept too, C folded into the next A: at most one slice a warp (117k rows
//     in FP64, 156k in FP32); the product gathers z + beta p
//   matrix kept: to 380k rows in FP64, 725k in FP32; its values stay off L2
//   vectors kept, matrix from L2 one slice ahead: to 1.1M rows in FP64, 2.2M in FP32
//   r and q kept (FP64): to 2.2M rows
// us an iteration (streaming kernels, then this): 32^3 FP64 19.7 -> 6.8, 97x61x83 FP32
// 32.6 -> 9.1, 64^3 FP64 34.5 -> 13.5, 128^3 FP64 91.7 -> 61.9, 128^3 FP32 on 8 parts
// 51.4 -> 31.4.
//
// The barrier is an arrival counter in L2 (red.release, ld.acquire polls of one
// thread a block): 1.3 us on 152 SMs. (Flags with the partial sums as payload took
// 5400 to 6700 cycles a sum with any number of replicas polled: the polls delay the
// writes they wait for.) The launch is cooperative, so all blocks are resident; every
// wait is bounded by spin probes all the same and ends the solve with
// RP_DEVICE_TIMEOUT (limits too small for a meeting never get here: kResidentSpin).
//
// Bound: small systems by the meetings (4000 cycles a sum, 2600 the barrier) and the
// latency of the gathers; FP32 at 2M rows by the products' instructions; FP64 at 128^3
// by the FP64 pipe (14 instructions a row and iteration with z kept, where K2 and K3
// compute it twice; the pipe 75% busy).
#include "rp_pcg.cuh"

namespace rp {
namespace {

// The run's scalars, the same in every block: thread 0's alone (in registers of
// every thread they spill the slice fetched ahead). alpha, beta: what all threads
// read. stop 2: before the x update, 3: at the cap.
template <typename T>
struct RsShared : RsFlags {
  T alpha, beta;
  double pq, rz, rr;
  int iter, iter_total, status, done;
  int unit[3];  // of (p, q), (r, z) and (r, r)
};

// LAY: layout of the product; SCALED: the system S A S (z = r); ALL: r, x, p
// and q in shared memory, else r and q; MAT: the matrix too; FOLD: no barrier C (the
// product gathers z + beta p of the two vectors, which are written to global memory
// before the sum of B).
template <typename T, int LAY, bool SCALED, bool ALL, bool MAT, bool FOLD>
__global__ void __launch_bounds__(kRsThreads<T, MAT>, 1) k_resident(const ResidentArgs<T> A) {
  const IterArgs<T>& a = A.it;
  Ctl* c = a.ctl;
  // written again only after every block has arrived once (or given up)
  if (c->stop || c->status == RP_DEVICE_TIMEOUT) return;
  extern __shared__ __align__(128) unsigned char sbuf[];
  __shared__ RsShared<T> sh;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nw = blockDim.x >> 5;
  T* rs = reinterpret_cast<T*>(sbuf);
  T* qs = rs + A.rows;
  T* ps = qs + A.rows;
  T* xs = ps + A.rows;
  T* xg = a.xd;
  if (xg == nullptr) xg = reinterpret_cast<T*>(a.io->x);

  RsBarrier bar{A.sync + kRsCount, A.sync[kRsBase], A.spin};
  int set = (int)A.sync[kRsSet];  // accumulators of this iteration's sums
  const double thresh = a.xd ? c->inner_thresh : c->thresh;
  const int max_iter = c->max_iter;
  if (tid == 0) {
    sh.pq = 0.0;
    sh.rz = c->rz;
    sh.rr = c->rr;
    sh.iter = c->iter;
    sh.iter_total = c->iter_total;
    sh.status = c->status;
    sh.bad = sh.stop = sh.done = sh.over = 0;
    for (int k = 0; k < 3; ++k) sh.unit[k] = (int)A.sync[kRsUnit + k];
  }
  using Matrix = RsMatrix<T, LAY, MAT>;
  static_assert(!FOLD || (ALL && Matrix::U4), "folded: p on chip, any row gathered by a functor");
  Matrix M(a.sl, a.parts, a.row_ptr, a.col, a.vals, (int)a.n,
           reinterpret_cast<unsigned char*>(rs + (ALL ? 4 : 2) * (size_t)A.rows), A.rows / 32, A.width);
  const int cnt = M.cnt;
  // FOLD: z, the last p and where it goes next; the first p is in memory as it is
  T* const zbuf = SCALED ? a.r : a.q;
  T* pcur = a.p;
  const T *zg = a.p, *pold = a.p;
  T fold_beta = T(0);
  for (int j = w; j < cnt; j += nw) {
    const int i = M.row_of(j), k = j * 32 + lane;
    rs[k] = i >= 0 ? a.r[i] : T(0);
    qs[k] = T(0);
    if (ALL) {
      ps[k] = i >= 0 ? a.p[i] : T(0);
      xs[k] = i >= 0 ? xg[i] : T(0);
    }
  }
  constexpr int W = ALL ? 16 / (int)sizeof(T) : 1;  // rows a thread takes at once outside the product
  __syncthreads();

  double* part = a.partials;  // two sets of partial sums in turn
  double* part2 = a.partials + 2 * (size_t)gridDim.x;
  for (;;) {
    // A: q = A p, (p, q)
    T acc = T(0);
    auto gathers = [&] {
      if constexpr (FOLD) return RsFold<T>{zg, pold, fold_beta};
      else return RsGlobal<T>{a.p};
    };
    const auto from = gathers();
    for (int j = w; j < cnt; j += nw) {
      const int i = M.row_of(j), k = j * 32 + lane;
      const T sum = M.product(j, i, from);
      if (i >= 0) {
        qs[k] = sum;
        acc = fma(ALL ? ps[k] : a.p[i], sum, acc);
      }
    }
    {
      const T v[1] = {acc};
      grid_sum_unit<1, false>(v, sh.unit, rs_words(A.sync, set, 0), sh, bar, part, lane, w, nw, [&](const double (&tot)[1]) {
        if (lane != 0) return;
        sh.pq = tot[0];
        sh.alpha = ratio<T>(sh.rz, tot[0]);
        if (!(tot[0] > 0.0) || !isfinite(tot[0])) {
          sh.status = RP_BREAKDOWN;
          sh.stop = 2;
        }
      });
    }
    if (sh.bad || sh.stop) break;
    // every block has left the sums of the iteration before: their accumulators are
    // cleared for the one after the next (seen by all behind barrier C)
    const int free_set = set == 0 ? 2 : set - 1;
    if (blockIdx.x == 0 && tid < 8) rs_words(A.sync, free_set, 0)[tid] = 0ull;  // two sums
    // B: r -= alpha q, z = D^-1 r (kept in q's place), x += alpha p, (r, z), (r, r)
    const T alpha = sh.alpha;
    T rza = T(0), rra = T(0);
    M.template groups<W>([&](int k, int i, int m, bool whole) {
      const RsPack<T, W> q = ld_pack<W>(qs + k);
      RsPack<T, W> r = ld_pack<W>(rs + k);
#pragma unroll
      for (int e = 0; e < W; ++e) {
        r.e[e] = fma(-alpha, q.e[e], r.e[e]);
        rra = fma(r.e[e], r.e[e], rra);
      }
      st_pack<W>(rs + k, r);
      if constexpr (SCALED && FOLD) st_rows<W>(zbuf + i, r, m, whole);
      if constexpr (!SCALED) {
        RsPack<T, W> z = ld_rows<W, true>(a.dinv + i, m, whole);
#pragma unroll
        for (int e = 0; e < W; ++e) {
          z.e[e] *= r.e[e];
          rza = fma(r.e[e], z.e[e], rza);
        }
        st_pack<W>(qs + k, z);
        if constexpr (FOLD) st_rows<W>(zbuf + i, z, m, whole);
      }
      if constexpr (ALL) {
        const RsPack<T, W> pv = ld_pack<W>(ps + k);
        RsPack<T, W> x = ld_pack<W>(xs + k);
#pragma unroll
        for (int e = 0; e < W; ++e) x.e[e] = fma(alpha, pv.e[e], x.e[e]);
        st_pack<W>(xs + k, x);
      } else {
        xg[i] = fma(alpha, a.p[i], xg[i]);
      }
    });
    {
      constexpr int NV = SCALED ? 1 : 2;
      T v[NV];
      v[NV - 1] = rra;
      if constexpr (!SCALED) v[0] = rza;
      grid_sum_unit<NV, FOLD>(v, sh.unit + 1, rs_words(A.sync, set, 1), sh, bar, part2, lane, w, nw, [&](const double (&tot)[NV]) {
        if (lane != 0) return;
        sh.rr = tot[NV - 1];
        ++sh.iter;
        ++sh.iter_total;
        ++sh.done;
        if (sh.rr <= thresh || sh.iter >= max_iter) {
          sh.stop = 1;
        } else if (!(tot[0] > 0.0) || !isfinite(tot[0])) {
          sh.stop = 1;
          sh.status = RP_BREAKDOWN;
        } else {
          sh.beta = ratio<T>(tot[0], sh.rz);
          sh.rz = tot[0];
          if (sh.done >= A.cap) sh.stop = 3;  // after C; the next launch goes on
        }
      });
    }
    set = set == 2 ? 0 : set + 1;
    if (sh.bad || sh.stop == 1) break;
    // C: p = z + beta p
    const T beta = sh.beta;
    T* const pnext = !FOLD || pcur != a.p ? a.p : SCALED ? a.q : a.r;
    M.template groups<W>([&](int k, int i, int m, bool whole) {
      RsPack<T, W> p;
      if constexpr (ALL) p = ld_pack<W>(ps + k);
      else p.e[0] = a.p[i];
      const RsPack<T, W> z = ld_pack<W>((SCALED ? rs : qs) + k);
#pragma unroll
      for (int e = 0; e < W; ++e) p.e[e] = fma(beta, p.e[e], z.e[e]);
      if constexpr (ALL) st_pack<W>(ps + k, p);
      st_rows<W>(pnext + i, p, m, whole);
    });
    __syncthreads();
    if constexpr (FOLD) {
      zg = zbuf;
      pold = pcur;
      pcur = pnext;
      fold_beta = beta;
    } else {
      if (tid == 0 && !bar.meet()) sh.bad = 1;
      __syncthreads();
    }
    if (sh.bad || sh.stop) break;
  }
  // the state back to memory (without FOLD p is there already)
  __syncthreads();
  for (int j = w; j < cnt; j += nw) {
    const int i = M.row_of(j), k = j * 32 + lane;
    if (i < 0) continue;
    a.r[i] = rs[k];
    if (ALL) xg[i] = xs[k];
    if (FOLD) a.p[i] = ps[k];
  }
  if (blockIdx.x == 0 && tid == 0) {
    A.sync[kRsBase] = bar.target;
    A.sync[kRsSet] = (unsigned int)set;
    for (int k = 0; k < 3; ++k) A.sync[kRsUnit + k] = (unsigned int)sh.unit[k];
    c->iter = sh.iter;
    c->iter_total = sh.iter_total;
    c->pq = sh.pq;
    c->rz = sh.rz;
    c->rr = sh.rr;
    atomicMax(&c->status, sh.status);  // a timeout, the largest status, stands whoever writes last
    if (sh.stop != 3) c->stop = 1;  // 0 at the launch and only ever raised: another block's report stands
    if (sh.stop == 2) c->skip_x = 1;
  }
  if (tid == 0 && sh.bad) {  // any block may have given up
    atomicMax(&c->status, (int)RP_DEVICE_TIMEOUT);
    c->stop = 1;
  }
}

template <typename T, bool ALL>
void* streamed_fn(int lay, bool scaled) {
  if constexpr (sizeof(T) == 4) {
    if (scaled)
      return lay == kRsU4 ? (void*)k_resident<T, kRsU4, true, ALL, false, false>
                          : (void*)k_resident<T, kRsSliced, true, ALL, false, false>;
  }
  switch (lay) {
    case kRsU4: return (void*)k_resident<T, kRsU4, false, ALL, false, false>;
    case kRsSliced: return (void*)k_resident<T, kRsSliced, false, ALL, false, false>;
    case kRsParts: return (void*)k_resident<T, kRsParts, false, ALL, false, false>;
    case kRsPartsU4: return (void*)k_resident<T, kRsPartsU4, false, ALL, false, false>;
    default: return (void*)k_resident<T, kRsCsr, false, ALL, false, false>;
  }
}
template <typename T, bool FOLD>
void* kept_fn(int lay, bool scaled) {
  if constexpr (sizeof(T) == 4) {
    if (scaled) return lay == kRsU4 ? (void*)k_resident<T, kRsU4, true, true, true, FOLD> : nullptr;
    return lay == kRsPartsU4 ? (void*)k_resident<T, kRsPartsU4, false, true, true, FOLD> : nullptr;
  } else {
    return lay == kRsU4        ? (void*)k_resident<T, kRsU4, false, true, true, FOLD>
           : lay == kRsPartsU4 ? (void*)k_resident<T, kRsPartsU4, false, true, true, FOLD>
                               : nullptr;
  }
}

}  // namespace

RP_CHECK_TU(resident)

// The forms, best first. Folding doubles the product's gathers to save a barrier: only
// where a warp has one slice.
enum : int { kKeptFold, kKept, kStream4, kStream2 };
template <typename T>
constexpr int kFoldRows = kRsThreads<T, true>;
template <typename T>
ResidentPlan resident_plan(const rp_handle* h, const IterArgs<T>& a, bool scaled) {
  if (a.line.l != nullptr) return ResidentPlan{};
  auto fn = [&](int lay, const ResidentForm& f) -> void* {
    if constexpr (sizeof(T) == 8)
      if (f.id == kStream2) return streamed_fn<T, false>(lay, scaled);
    if (f.id == kKept) return kept_fn<T, false>(lay, scaled);
    return f.id == kKeptFold ? kept_fn<T, true>(lay, scaled) : streamed_fn<T, true>(lay, scaled);
  };
  constexpr int64_t kL2 = 80'000'000;
  constexpr ResidentForm kFold{4, true, kFoldRows<T>, kKeptFold, RP_FORM_RESIDENT_FOLDED};
  constexpr ResidentForm kMat{4, true, INT32_MAX, kKept, RP_FORM_RESIDENT_MATRIX};
  constexpr ResidentForm kFour{4, false, INT32_MAX, kStream4}, kTwo{2, false, INT32_MAX, kStream2};
  if constexpr (sizeof(T) == 8) return plan_resident<T>(h, a.sl, a.n, kL2, {kFold, kMat, kFour, kTwo}, fn);
  else return plan_resident<T>(h, a.sl, a.n, kL2, {kFold, kMat, kFour}, fn);
}
template ResidentPlan resident_plan<double>(const rp_handle*, const IterArgs<double>&, bool);
template ResidentPlan resident_plan<float>(const rp_handle*, const IterArgs<float>&, bool);

}  // namespace rp
