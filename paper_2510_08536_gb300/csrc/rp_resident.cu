// The resident form of the PCG iteration: one cooperative launch (one block an
// SM) runs a whole inner run, with the vectors in shared memory.
//
// The streaming form (K1, K2, K3 of rp_pcg.cu in a conditional graph) costs
// 20 us an iteration however small the system is: three launches, two block
// elections and the latency of cold pipelines. Systems whose vectors fit the
// SMs' shared memory (152 x 227 KB) need none of it: block b owns a contiguous
// run of 32-row slices and keeps r, x, p and q of those rows in shared memory
// (FP64 beyond 7,200 rows an SM: r and q); only p, which the products gather
// across blocks, is also written to global memory, and the matrix streams from
// L2. The grid meets three times an iteration:
//   A  q = A p,                             (p, q)          | sum -> alpha
//   B  r -= alpha q, z = D^-1 r, x += alpha p, (r, z), (r, r) | sum -> beta, stop test
//   C  p = z + beta p                                       | barrier
// with the arithmetic of K1-K3, row by row the same fused multiply-adds; the
// dot products are summed per thread, warp and block and over the blocks in
// block order (rp_reduce.cuh), every block summing all partials itself, so all
// blocks hold the same scalars and take the same branches.
//
// The barrier is an arrival counter in L2 (red.release, ld.acquire polls of one
// thread a block): 1.3 us on 152 SMs. (Flags with the partial sums as payload,
// polled by all blocks, took 5-8 us: the polls delay the writes they wait for.)
// The launch is cooperative, so all blocks are resident; every wait is bounded
// by spin probes all the same and ends the solve with RP_DEVICE_TIMEOUT.
//
// Bound: small systems by the three meetings and the latency of the gathers;
// FP64 at 128^3 by the FP64 pipe (14 instructions a row and iteration with z
// kept, where K2 and K3 compute it twice).
#include <algorithm>

#include "rp_common.cuh"
#include "rp_pcg.cuh"
#include "rp_spmv.cuh"

namespace rp {
namespace {

// layouts of the product: CSR, sliced, sliced and uniform (4-bit indices, rows
// of at most 8 entries), and both with several parts
enum : int { kRsCsr = 0, kRsSliced = 1, kRsU4 = 2, kRsParts = 3, kRsPartsU4 = 4 };

// FP64: 24 warps of up to 80 registers (32 warps of 64 spill the prefetched
// slice, and the FP64 pipe is the bound anyway)
template <typename T>
constexpr int kRsThreads = sizeof(T) == 8 ? 768 : 1024;

// Scalars every thread needs, written by warp 0 between the two block barriers
// of a grid sum.
template <typename T>
struct RsShared {
  double warp[2][32];
  T alpha, beta;
  int stop;  // leave the loop; 2: before the x update
  int bad;   // a wait ran out
};

// One block's arrival at the grid barrier and its wait for all others (one
// thread; the block's earlier writes are released, the others' acquired).
struct RsBarrier {
  unsigned int* cnt;
  unsigned int target;
  int64_t spin;
  __device__ __forceinline__ bool meet() {
    target += gridDim.x;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(cnt) : "memory");
    for (int64_t i = 0; i < spin; ++i) {
      unsigned int v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(cnt) : "memory");
      if ((int)(v - target) >= 0) return true;
    }
    return false;
  }
};

// Grid sum of NV values a thread. Warp 0 of every block receives the totals in
// tot[] (all lanes) and calls fin(tot, ok); then the block goes on together.
template <int NV, typename T, typename Fin>
__device__ __forceinline__ void grid_sum(const T (&v)[NV], RsShared<T>& sh, RsBarrier& bar, double* partials, int lane,
                                         int w, int nw, Fin&& fin) {
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const double s = warp_sum(v[i]);
    if (lane == 0) sh.warp[i][w] = s;
  }
  __syncthreads();
  if (w == 0) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const double s = warp_sum(lane < nw ? sh.warp[i][lane] : 0.0);
      if (lane == 0) __stcg(partials + (size_t)blockIdx.x * NV + i, s);
    }
    int ok = 1;
    if (lane == 0) ok = bar.meet() ? 1 : 0;
    ok = __shfl_sync(0xffffffffu, ok, 0);
    __syncwarp();
    constexpr int kPer = 5;  // 160 blocks a trip: one trip on 152 SMs
    double tot[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      double s = 0.0;
      for (unsigned int b0 = 0; b0 < gridDim.x; b0 += 32 * kPer) {
        double x[kPer];
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
          const unsigned int b = b0 + 32 * j + lane;
          x[j] = b < gridDim.x ? __ldcg(partials + (size_t)b * NV + i) : 0.0;
        }
        const double t = warp_sum_n(x);
        s = b0 ? s + t : t;
      }
      tot[i] = s;
    }
    if (lane == 0 && !ok) sh.bad = 1;
    fin(tot);
  }
  __syncthreads();
}

// read-only data of one pass an iteration: not worth a line of L1
__device__ __forceinline__ float ldg_stream(const float* p) {
  float v;
  asm volatile("ld.global.nc.L1::no_allocate.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ double ldg_stream(const double* p) {
  double v;
  asm volatile("ld.global.nc.L1::no_allocate.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ uint32_t ldg_stream(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.global.nc.L1::no_allocate.u32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}

// A slice of the uniform layout (4-bit indices, at most 8 entries a row) held
// in registers: loaded one slice ahead, across the grid barriers too, so that
// only the gathers of p wait on memory.
template <typename T>
struct RsSlice {
  T v[8];
  uint32_t wd;
  int32_t tv;
  int L;
  __device__ __forceinline__ void load(const Sliced<T>& sl, uint2 d0, uint2 d1, uint32_t info, int lane) {
    L = (int)((d1.x - d0.x) >> 5);
    const T* p = sl.vals + d0.x + lane;
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (k < L) v[k] = ldg_stream(p + 32 * k);
    wd = L > 0 ? ldg_stream(reinterpret_cast<const uint32_t*>(sl.ibuf) + d0.y + lane) : 0u;
    tv = __ldg(sl.tabs + (info & ~kSliceW4) + (lane & 15));
  }
  // the row's products in entry order; x: the gathered vector at the lane's row
  __device__ __forceinline__ T sum(const T* x, bool valid) const {
    T g[8];
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (k < L) {
        const int off = slice_offset<kIdx4>(wd, k, tv, nullptr, 0);
        g[k] = valid ? x[off] : T(0);
      }
    T s = T(0);
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (k < L) s = fma(v[k], g[k], s);
    return s;
  }
};

// LAY: layout of the product; SCALED: the system S A S (z = r); ALL: r, x, p
// and q in shared memory, else r and q.
template <typename T, int LAY, bool SCALED, bool ALL>
__global__ void __launch_bounds__(kRsThreads<T>, 1) k_resident(const ResidentArgs<T> A) {
  constexpr bool MP = LAY == kRsParts || LAY == kRsPartsU4, U4 = LAY == kRsU4 || LAY == kRsPartsU4;
  const IterArgs<T>& a = A.it;
  Ctl* c = a.ctl;
  // written again only after every block has arrived once (or given up)
  if (c->stop || c->status == RP_DEVICE_TIMEOUT) return;
  extern __shared__ __align__(128) unsigned char sbuf[];
  __shared__ RsShared<T> sh;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nw = blockDim.x >> 5;
  const int n = (int)a.n;
  const int S = LAY == kRsCsr ? (n + 31) / 32 : (int)a.sl.n_slices;
  const int s0 = (int)((int64_t)S * blockIdx.x / gridDim.x);
  const int cnt = (int)((int64_t)S * (blockIdx.x + 1) / gridDim.x) - s0;
  T* rs = reinterpret_cast<T*>(sbuf);
  T* qs = rs + A.rows;
  T* ps = qs + A.rows;
  T* xs = ps + A.rows;
  unsigned char* tail = reinterpret_cast<unsigned char*>(rs + (ALL ? 4 : 2) * (size_t)A.rows);
  uint2* sdesc = reinterpret_cast<uint2*>(tail);  // [cnt + 1]
  int2* srow = reinterpret_cast<int2*>(sdesc + A.rows / 32 + 1);
  uint32_t* sinfo = reinterpret_cast<uint32_t*>(srow + (MP ? A.rows / 32 : 0));
  int32_t* snl = reinterpret_cast<int32_t*>(sinfo + A.rows / 32);  // MP: first non-local entry of the slice's part
  T* xg = a.xd;
  if (xg == nullptr) xg = reinterpret_cast<T*>(a.io->x);

  RsBarrier bar{A.sync, A.sync[32], A.spin};
  // scalars of the run: kept by warp 0, the same in every block
  double rz = c->rz, rr = c->rr, pq = 0.0;
  const double thresh = a.xd ? c->inner_thresh : c->thresh;
  int iter = c->iter, iter_total = c->iter_total, status = c->status, done = 0;
  const int max_iter = c->max_iter;
  if (tid == 0) sh.bad = sh.stop = 0;
  if (LAY != kRsCsr) {
    for (int j = tid; j <= cnt; j += blockDim.x) sdesc[j] = a.sl.desc[s0 + j];
    for (int j = tid; j < cnt; j += blockDim.x) {
      sinfo[j] = a.sl.tinfo[s0 + j];
      if (MP) {
        const int2 r = a.sl.srow[s0 + j];
        srow[j] = r;
        snl[j] = (int32_t)a.parts.nl_off[r.y >> 6];
      }
    }
  }
  __syncthreads();
  // row of slice j for this lane, or -1
  auto row_of = [&](int j) -> int {
    if (MP) {
      const int2 r = srow[j];
      return lane < (r.y & 63) ? r.x + lane : -1;
    }
    const int i = (s0 + j) * kSliceRows + lane;
    return i < n ? i : -1;
  };
  for (int j = w; j < cnt; j += nw) {
    const int i = row_of(j), k = j * 32 + lane;
    if (i < 0) continue;
    rs[k] = a.r[i];
    if (ALL) {
      ps[k] = a.p[i];
      xs[k] = xg[i];
    }
  }
  RsSlice<T> f;
  NlRange fnl{0, 0};
  auto fetch = [&](int j) {
    f.load(a.sl, sdesc[j], sdesc[j + 1], sinfo[j], lane);
    if (MP) {
      const int i = row_of(j);
      fnl = i >= 0 ? nonlocal_range<T>(a.parts, srow[j].y >> 6, i) : NlRange{0, 0};
    }
  };
  if (U4 && w < cnt) fetch(w);

  double* part = a.partials;  // two sets of partial sums in turn
  double* part2 = a.partials + 2 * (size_t)gridDim.x;
  for (;;) {
    // A: q = A p, (p, q)
    T acc = T(0);
    for (int j = w; j < cnt; j += nw) {
      const int i = row_of(j), k = j * 32 + lane;
      const bool valid = i >= 0;
      T sum = T(0);
      if constexpr (U4) {
        const RsSlice<T> cur = f;
        const NlRange nl = fnl;
        fetch(j + nw < cnt ? j + nw : w);  // the last one fetches the first of the next iteration
        int g = 0;
        T gv = T(0);
        const int nlo = MP ? snl[j] : 0;
        if (MP && nl.j0 < nl.j1) {  // the first non-local entry alongside the gathers
          g = __ldg(a.parts.nl_gcol + nlo + nl.j0);
          gv = __ldg(a.parts.nl_vals + nlo + nl.j0);
        }
        sum = cur.sum(a.p + (valid ? i : 0), valid);
        if (MP && nl.j0 < nl.j1) {
          sum = fma(gv, a.p[g], sum);
          for (int e = nl.j0 + 1; e < nl.j1; ++e)
            sum = fma(__ldg(a.parts.nl_vals + nlo + e), a.p[__ldg(a.parts.nl_gcol + nlo + e)], sum);
        }
      } else if constexpr (LAY == kRsCsr) {
        if (valid) sum = row_dot_any<T, true>(a.parts, a.row_ptr, a.col, a.vals, a.p, i, n);
      } else {
        const int part_id = MP ? srow[j].y >> 6 : 0;
        NlRange nl{0, 0};
        if constexpr (MP)
          if (valid) nl = nonlocal_range<T>(a.parts, part_id, i);
        const SliceCk ck = slice_ck<T, MP>(a.sl, a.parts, part_id, i, n);
        const uint2 d0 = sdesc[j], d1 = sdesc[j + 1];
        sum = slice_sum<T, true>(d0, d1, sinfo[j], a.sl.vals + d0.x + lane,
                                 reinterpret_cast<const uint32_t*>(a.sl.ibuf) + d0.y + lane, a.sl.tabs,
                                 a.p + (valid ? i : 0), valid, lane, ck);
        if constexpr (MP)
          if (valid) sum = nonlocal_sum<T, true>(a.parts, part_id, nl, a.p, sum);
      }
      if (valid) {
        qs[k] = sum;
        acc = fma(ALL ? ps[k] : a.p[i], sum, acc);
      }
    }
    {
      const T v[1] = {acc};
      grid_sum<1>(v, sh, bar, part, lane, w, nw, [&](const double (&tot)[1]) {
        pq = tot[0];
        const bool broke = !(pq > 0.0) || !isfinite(pq);
        if (broke) status = RP_BREAKDOWN;
        const T alpha = (T)(rz / pq);
        if (lane == 0) {
          sh.alpha = alpha;
          if (broke) sh.stop = 2;
        }
      });
    }
    if (sh.bad || sh.stop) break;
    // B: r -= alpha q, z = D^-1 r (kept in q's place), x += alpha p, (r, z), (r, r)
    const T alpha = sh.alpha;
    T rza = T(0), rra = T(0);
    for (int j = w; j < cnt; j += nw) {
      const int i = row_of(j), k = j * 32 + lane;
      if (i < 0) continue;
      const T ri = fma(-alpha, qs[k], rs[k]);
      rs[k] = ri;
      if (!SCALED) {
        const T z = a.dinv[i] * ri;
        qs[k] = z;
        rza = fma(ri, z, rza);
      }
      rra = fma(ri, ri, rra);
      if (ALL) xs[k] = fma(alpha, ps[k], xs[k]);
      else xg[i] = fma(alpha, a.p[i], xg[i]);
    }
    {
      constexpr int NV = SCALED ? 1 : 2;
      T v[NV];
      v[NV - 1] = rra;
      if constexpr (!SCALED) v[0] = rza;
      grid_sum<NV>(v, sh, bar, part2, lane, w, nw, [&](const double (&tot)[NV]) {
        const double rzn = tot[0];
        rr = tot[NV - 1];
        ++iter;
        ++iter_total;
        ++done;
        int stop = 0;
        if (rr <= thresh || iter >= max_iter) {
          stop = 1;
        } else if (!(rzn > 0.0) || !isfinite(rzn)) {
          stop = 1;
          status = RP_BREAKDOWN;
        } else {
          const T beta = (T)(rzn / rz);
          if (lane == 0) sh.beta = beta;
          rz = rzn;
        }
        if (lane == 0) sh.stop = stop;
      });
    }
    if (sh.bad || sh.stop) break;
    // C: p = z + beta p
    const T beta = sh.beta;
    for (int j = w; j < cnt; j += nw) {
      const int i = row_of(j), k = j * 32 + lane;
      if (i < 0) continue;
      const T pi = fma(beta, ALL ? ps[k] : a.p[i], SCALED ? rs[k] : qs[k]);
      if (ALL) ps[k] = pi;
      a.p[i] = pi;
    }
    __syncthreads();
    if (tid == 0) {
      if (!bar.meet()) sh.bad = 1;
      if (done >= A.cap) sh.stop = 3;  // the next launch goes on
    }
    __syncthreads();
    if (sh.bad || sh.stop) break;
  }
  // the state back to memory (p is there already)
  for (int j = w; j < cnt; j += nw) {
    const int i = row_of(j), k = j * 32 + lane;
    if (i < 0) continue;
    a.r[i] = rs[k];
    if (ALL) xg[i] = xs[k];
  }
  if (blockIdx.x == 0 && tid == 0) {
    A.sync[32] = bar.target;
    c->iter = iter;
    c->iter_total = iter_total;
    c->pq = pq;
    c->rz = rz;
    c->rr = rr;
    atomicMax(&c->status, status);  // a timeout, the largest status, stands whoever writes last
    c->stop = sh.stop == 3 ? 0 : 1;
    if (sh.stop == 2) c->skip_x = 1;
  }
  if (tid == 0 && sh.bad) {  // any block may have given up
    atomicMax(&c->status, (int)RP_DEVICE_TIMEOUT);
    c->stop = 1;
  }
}

template <typename T, bool ALL>
void* resident_fn(int lay, bool scaled) {
  if constexpr (sizeof(T) == 4) {
    if (scaled)
      return lay == kRsU4 ? (void*)k_resident<T, kRsU4, true, ALL> : (void*)k_resident<T, kRsSliced, true, ALL>;
  }
  switch (lay) {
    case kRsU4: return (void*)k_resident<T, kRsU4, false, ALL>;
    case kRsSliced: return (void*)k_resident<T, kRsSliced, false, ALL>;
    case kRsParts: return (void*)k_resident<T, kRsParts, false, ALL>;
    case kRsPartsU4: return (void*)k_resident<T, kRsPartsU4, false, ALL>;
    default: return (void*)k_resident<T, kRsCsr, false, ALL>;
  }
}

}  // namespace

RP_CHECK_TU(resident)

template <typename T>
ResidentPlan resident_plan(const rp_handle* h, const IterArgs<T>& a, bool scaled) {
  ResidentPlan p;
  int coop = 0, smem_max = 0;
  if (a.line.l != nullptr || a.n == 0) return p;
  if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, h->device) != cudaSuccess || !coop ||
      cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, h->device) != cudaSuccess) {
    cudaGetLastError();
    return p;
  }
#ifdef RP_CHECK
  const bool u4 = false;  // the checked build tests every slice
#else
  const bool u4 = a.sl.u4 != 0;
#endif
  const int lay = a.sl.n_slices == 0 ? kRsCsr : a.sl.srow ? (u4 ? kRsPartsU4 : kRsParts) : u4 ? kRsU4 : kRsSliced;
  const int64_t S = lay == kRsCsr ? (a.n + 31) / 32 : a.sl.n_slices;
  const int grid = (int)std::min<int64_t>(h->num_sms, S);
  const int64_t per = (S + grid - 1) / grid;  // slices a block at most
  const int64_t tail = lay == kRsCsr ? 0 : (per + 1) * 8 + per * 4 + (a.sl.srow ? per * 12 : 0);
  // the kernel's own (static) shared memory comes off the block's limit
  auto fits = [&](void* fn, int vecs) {
    const int64_t need = per * 32 * vecs * (int64_t)sizeof(T) + tail;
    const int threads = 32 * (int)std::min<int64_t>(std::max<int64_t>(per, 4), kRsThreads<T> / 32);
    cudaFuncAttributes at;
    int nb = 0;
    if (cudaFuncGetAttributes(&at, fn) != cudaSuccess || need > smem_max - (int)at.sharedSizeBytes ||
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max - (int)at.sharedSizeBytes) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, threads, (size_t)need) != cudaSuccess || nb < 1) {
      cudaGetLastError();
      return false;
    }
    p = ResidentPlan{fn, grid, threads, (int)need, (int)(per * 32)};
    return true;
  };
  if (fits(resident_fn<T, true>(lay, scaled), 4)) return p;
  if constexpr (sizeof(T) == 8) fits(resident_fn<T, false>(lay, scaled), 2);
  return p;
}
template ResidentPlan resident_plan<double>(const rp_handle*, const IterArgs<double>&, bool);
template ResidentPlan resident_plan<float>(const rp_handle*, const IterArgs<float>&, bool);

}  // namespace rp
