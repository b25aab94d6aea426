// The resident form of the BiCGStab inner loop: one cooperative launch (one
// block an SM) runs every iteration, with four vectors in shared memory.
//
// The streaming form (B1-B5 of rp_bicgstab.cu in a conditional graph) makes five
// launches and three block elections an iteration and moves every vector through
// L2 between them. Here block b owns a contiguous run of 32-row slices and keeps
// p, v, t and r (s in its place between B3 and B5) of those rows in shared
// memory; phat and shat, which the products gather across blocks, are also
// written to global memory, and their own rows recomputed as D^-1 p and D^-1 s;
// rhat, x, D^-1 and the matrix are read from L2. The grid meets five times an
// iteration:
//   B1  p = r + beta (p - omega v), phat           | barrier
//   B2  v = A phat, (rhat, v)                      | sum -> alpha
//   B3  s = r - alpha v, shat, (s, s)              | sum -> half step
//   B4  t = A shat, (t, s), (t, t)                 | sum -> omega
//   B5  x += alpha phat + omega shat, r = s - omega t, (r, r), (rhat, r) | sum -> beta, stop
// with the fused multiply-adds of B1-B5 row by row. Barriers and sums are those
// of rp_resident.cuh; every wait is bounded and ends the solve with
// RP_DEVICE_TIMEOUT.
//
// 128^3 mixed, a momentum step of 214 iterations: 26.0 ms with the streaming kernels,
// 14.5 ms with this one and sums by way of all blocks' partial sums, 13.9 ms with sums
// in known units, 12.1 ms with 28 warps that do not spill. Bound: the products'
// instructions and the five meetings; in FP64 the FP64 pipe (28 instructions a row and iteration).
#include "rp_bicgstab.cuh"

namespace rp {
namespace {

// The run's scalars, the same in every block: thread 0's alone (registers of
// every thread would spill the slice fetched ahead). al, om, be: what all threads
// read. stop 2: the cap; 3: half step (leaves after its x update).
template <typename T>
struct BsShared : RsFlags {
  T al, om, be;
  double rho, rho_old, alpha, omega, rr, ss;
  int iter, status, done;
  int unit[6];  // of (rhat, v), (s, s), (t, s), (t, t), (r, r), (rhat, r)
};

template <typename T>
__device__ __forceinline__ const BsVecs<T>& vecs_of(const BsArgs& a) {
  if constexpr (sizeof(T) == 8) return a.d;
  else return a.f;
}

template <typename T, int LAY>
__global__ void __launch_bounds__(kRsThreads<T, false>, 1) k_resident_bs(const ResidentBsArgs<T> A) {
  const BsArgs& a = A.a;
  const BsVecs<T>& V = vecs_of<T>(a);
  BsCtl* c = a.c;
  // written again only after every block has arrived once (or given up)
  if (c->stop || c->status == RP_DEVICE_TIMEOUT) return;
  extern __shared__ __align__(128) unsigned char sbuf[];
  __shared__ BsShared<T> sh;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nw = blockDim.x >> 5;
  T* rs = reinterpret_cast<T*>(sbuf);
  T* ps = rs + A.rows;
  T* vs = ps + A.rows;
  T* ts = vs + A.rows;
  T* xg = V.x;
  if constexpr (sizeof(T) == 8) xg = a.io->x;
  const bool x16 = (reinterpret_cast<uintptr_t>(xg) & 15) == 0;  // the caller's may not be

  RsBarrier bar{A.sync + kRsCount, A.sync[kRsBase], A.spin};
  int set = (int)A.sync[kRsSet];  // accumulators of this iteration's sums
  const double thresh = c->ithresh;
  const int max_iter = c->max_iter;
  if (tid == 0) {
    sh.rho = c->rho;
    sh.rho_old = c->rho_old;
    sh.alpha = c->alpha;
    sh.omega = c->omega;
    sh.rr = c->rr;
    sh.ss = c->ss;
    sh.iter = c->iter;
    sh.status = c->status;
    sh.bad = sh.stop = sh.done = sh.over = 0;
    for (int k = 0; k < 6; ++k) sh.unit[k] = (int)A.sync[kRsUnit + k];
    sh.om = (T)sh.omega;
    sh.be = (T)((sh.rho / sh.rho_old) * (sh.alpha / sh.omega));
  }
  RsMatrix<T, LAY> M(V.sl, V.parts, a.row_ptr, a.col, V.vals, (int)a.n,
                     reinterpret_cast<unsigned char*>(ts + A.rows), A.rows / 32, 0);
  const int cnt = M.cnt;
  for (int j = w; j < cnt; j += nw) {
    const int i = M.row_of(j), k = j * 32 + lane;
    rs[k] = i >= 0 ? V.r[i] : T(0);
    ps[k] = i >= 0 ? V.p[i] : T(0);
    vs[k] = i >= 0 ? V.v[i] : T(0);
    ts[k] = T(0);
  }
  constexpr int W = 16 / (int)sizeof(T);  // rows a thread takes at once outside the products
  __syncthreads();

  double* part = a.partials;  // two sets of partial sums in turn
  double* part2 = a.partials + 2 * (size_t)gridDim.x;
  for (;;) {
    // B1
    {
      const T be = sh.be, om = sh.om;
      M.template groups<W>([&](int k, int i, int m, bool whole) {
        RsPack<T, W> p = ld_pack<W>(ps + k), h = ld_rows<W, true>(V.dinv + i, m, whole);
        const RsPack<T, W> v = ld_pack<W>(vs + k), r = ld_pack<W>(rs + k);
#pragma unroll
        for (int e = 0; e < W; ++e) {
          p.e[e] = fma(be, fma(-om, v.e[e], p.e[e]), r.e[e]);
          h.e[e] *= p.e[e];
        }
        st_pack<W>(ps + k, p);
        st_rows<W>(V.phat + i, h, m, whole);
      });
      __syncthreads();
      if (tid == 0 && !bar.meet()) sh.bad = 1;
      __syncthreads();
      if (sh.bad) break;
    }
    // B2
    {
      T acc = T(0);
      for (int j = w; j < cnt; j += nw) {
        const int i = M.row_of(j), k = j * 32 + lane;
        const T rh = i >= 0 ? __ldg(V.rhat + i) : T(0);
        const T y = M.product(j, i, RsGlobal<T>{V.phat});
        if (i >= 0) {
          vs[k] = y;
          acc = fma(rh, y, acc);
        }
      }
      const T v[1] = {acc};
      grid_sum_unit<1, false>(v, sh.unit, rs_words(A.sync, set, 0), sh, bar, part, lane, w, nw, [&](const double (&tot)[1]) {
        if (lane != 0) return;
        if (tot[0] == 0.0 || !isfinite(tot[0])) {
          sh.status = RP_BREAKDOWN;
          sh.stop = 1;
        } else {
          sh.alpha = quot_rn(sh.rho, tot[0]);
          sh.al = (T)sh.alpha;
        }
      });
    }
    if (sh.bad || sh.stop) break;
    // every block has left the sums of the iteration before: their accumulators are
    // cleared for the one after the next (seen by all behind the next barrier)
    if (blockIdx.x == 0 && tid < kRsSetWords) rs_words(A.sync, set == 0 ? 2 : set - 1, 0)[tid] = 0ull;
    const T al = sh.al;
    // B3
    {
      T acc = T(0);
      M.template groups<W>([&](int k, int i, int m, bool whole) {
        RsPack<T, W> r = ld_pack<W>(rs + k), h = ld_rows<W, true>(V.dinv + i, m, whole);
        const RsPack<T, W> v = ld_pack<W>(vs + k);
#pragma unroll
        for (int e = 0; e < W; ++e) {
          r.e[e] = fma(-al, v.e[e], r.e[e]);
          acc = fma(r.e[e], r.e[e], acc);
          h.e[e] *= r.e[e];
        }
        st_pack<W>(rs + k, r);
        st_rows<W>(V.shat + i, h, m, whole);
      });
      const T v[1] = {acc};
      grid_sum_unit<1, true>(v, sh.unit + 1, rs_words(A.sync, set, 1), sh, bar, part2, lane, w, nw, [&](const double (&tot)[1]) {
        if (lane != 0) return;
        sh.ss = tot[0];
        if (tot[0] <= thresh) sh.stop = 3;
      });
    }
    if (sh.bad) break;
    if (sh.stop == 3) {  // (the groups' rows are this block's: no wait since B1 is missing)
      for (int j = w; j < cnt; j += nw) {
        const int i = M.row_of(j), k = j * 32 + lane;
        if (i >= 0) xg[i] = fma(al, __ldg(V.dinv + i) * ps[k], xg[i]);
      }
      if (tid == 0) {
        ++sh.iter;
        sh.rr = sh.ss;
      }
      break;
    }
    // B4
    {
      T ats = T(0), att = T(0);
      for (int j = w; j < cnt; j += nw) {
        const int i = M.row_of(j), k = j * 32 + lane;
        const T y = M.product(j, i, RsGlobal<T>{V.shat});
        if (i >= 0) {
          ts[k] = y;
          ats = fma(y, rs[k], ats);
          att = fma(y, y, att);
        }
      }
      const T v[2] = {ats, att};
      grid_sum_unit<2, false>(v, sh.unit + 2, rs_words(A.sync, set, 2), sh, bar, part, lane, w, nw, [&](const double (&tot)[2]) {
        if (lane != 0) return;
        const double om = quot_rn(tot[0], tot[1]);
        if (!(tot[1] > 0.0) || !isfinite(om)) {
          sh.status = RP_BREAKDOWN;
          sh.stop = 1;
        } else {
          sh.omega = om;
          sh.om = (T)om;
        }
      });
    }
    if (sh.bad || sh.stop) break;
    // B5
    {
      const T om = sh.om;
      T arr = T(0), arh = T(0);
      M.template groups<W>([&](int k, int i, int m, bool whole) {
        RsPack<T, W> r = ld_pack<W>(rs + k);
        const RsPack<T, W> d = ld_rows<W, true>(V.dinv + i, m, whole), p = ld_pack<W>(ps + k), t = ld_pack<W>(ts + k);
        const RsPack<T, W> rh = ld_rows<W, true>(V.rhat + i, m, whole);
        const bool xw = whole && x16;
        RsPack<T, W> x = ld_rows<W, false>(xg + i, m, xw);
#pragma unroll
        for (int e = 0; e < W; ++e) {
          x.e[e] = fma(om, d.e[e] * r.e[e], fma(al, d.e[e] * p.e[e], x.e[e]));
          r.e[e] = fma(-om, t.e[e], r.e[e]);
          arr = fma(r.e[e], r.e[e], arr);
          arh = fma(rh.e[e], r.e[e], arh);
        }
        st_rows<W>(xg + i, x, m, xw);
        st_pack<W>(rs + k, r);
      });
      const T v[2] = {arr, arh};
      grid_sum_unit<2, false>(v, sh.unit + 4, rs_words(A.sync, set, 3), sh, bar, part2, lane, w, nw, [&](const double (&tot)[2]) {
        if (lane != 0) return;
        sh.rr = tot[0];
        ++sh.iter;
        int stop = ++sh.done >= A.cap ? 2 : 0;  // at the cap the next launch goes on
        if (tot[0] <= thresh || sh.iter >= max_iter) {
          stop = 1;
        } else if (sh.omega == 0.0 || tot[1] == 0.0 || !isfinite(tot[1])) {
          sh.status = RP_BREAKDOWN;
          stop = 1;
        } else {
          sh.rho_old = sh.rho;
          sh.rho = tot[1];
          sh.be = (T)(quot_rn(sh.rho, sh.rho_old) * quot_rn(sh.alpha, sh.omega));
        }
        sh.stop = stop;
      });
    }
    set = set == 2 ? 0 : set + 1;
    if (sh.bad || sh.stop) break;
  }
  if (sh.stop == 2) {  // the state back to memory for the next launch
    for (int j = w; j < cnt; j += nw) {
      const int i = M.row_of(j), k = j * 32 + lane;
      if (i < 0) continue;
      V.r[i] = rs[k];
      V.p[i] = ps[k];
      V.v[i] = vs[k];
    }
  }
  if (blockIdx.x == 0 && tid == 0) {
    A.sync[kRsBase] = bar.target;
    A.sync[kRsSet] = (unsigned int)(sh.stop == 3 ? (set == 2 ? 0 : set + 1) : set);
    for (int k = 0; k < 6; ++k) A.sync[kRsUnit + k] = (unsigned int)sh.unit[k];
    c->iter = sh.iter;
    c->rho = sh.rho;
    c->rho_old = sh.rho_old;
    c->alpha = sh.alpha;
    c->omega = sh.omega;
    c->rr = sh.rr;
    c->ss = sh.ss;
    c->half = sh.stop == 3;
    atomicMax(&c->status, sh.status);  // a timeout, the largest status, stands whoever writes last
    if (sh.stop != 2) c->stop = 1;  // 0 at the launch and only ever raised: another block's report stands
  }
  if (tid == 0 && sh.bad) {  // any block may have given up
    atomicMax(&c->status, (int)RP_DEVICE_TIMEOUT);
    c->stop = 1;
  }
}

}  // namespace

RP_CHECK_TU(resident_bs)

template <typename T>
ResidentPlan resident_bs_plan(const rp_handle* h, const BsVecs<T>& v) {
  return plan_resident<T>(h, v.sl, h->n, 75'000'000, {{4, false, INT32_MAX, 0}}, [](int lay, const ResidentForm&) -> void* {
    switch (lay) {
      case kRsU4: return (void*)k_resident_bs<T, kRsU4>;
      case kRsSliced: return (void*)k_resident_bs<T, kRsSliced>;
      case kRsParts: return (void*)k_resident_bs<T, kRsParts>;
      case kRsPartsU4: return (void*)k_resident_bs<T, kRsPartsU4>;
      default: return (void*)k_resident_bs<T, kRsCsr>;
    }
  });
}
template ResidentPlan resident_bs_plan<double>(const rp_handle*, const BsVecs<double>&);
template ResidentPlan resident_bs_plan<float>(const rp_handle*, const BsVecs<float>&);

}  // namespace rp
