// Building blocks of the resident solver kernels (rp_resident.cu: PCG,
// rp_resident_bs.cu: BiCGStab): one block an SM owns a contiguous run of 32-row
// slices, a warp takes every nw-th of them in the products and 16-byte groups of
// rows in the passes over vectors, and the grid meets at an arrival counter.
#pragma once

#include <algorithm>
#include <initializer_list>

#include "rp_common.cuh"
#include "rp_spmv.cuh"
#include "rp_values.cuh"

namespace rp {

// layouts of the product: CSR, sliced, sliced and uniform (4-bit indices, rows
// of at most 8 entries), and both with several parts
enum : int { kRsCsr = 0, kRsSliced = 1, kRsU4 = 2, kRsParts = 3, kRsPartsU4 = 4 };

// Threads of a block: as many as leave the slice fetched ahead its registers. FP32
// streamed, us an iteration at 128^3 (one part, 8 parts, BiCGStab): 32 warps of 64
// registers 34.1, 39.6, 62.0 (they spill); 28 of 72 25.9, 31.4, 52.3; 24 of 80 27.1,
// 34.4, 57.9; 16 of 128 lose more. With the matrix in shared memory 64 registers are
// enough for FP32. FP64 (28 instructions of its pipe a slice): 24 warps of 80.
template <typename T, bool MAT>
constexpr int kRsThreads = sizeof(T) == 8 ? 768 : MAT ? 1024 : 896;

// Partial sums of a block's warps, and the flags every thread reads after a grid sum.
struct RsFlags {
  union {
    double warp[2][32];
    uint32_t digit[2][kFixDigits][32];
  };
  int stop;  // leave the loop (each kernel's own codes)
  int bad;   // a wait ran out
  int over;  // a value past the range of its sum's unit
  int again; // the sum has to be taken from the blocks' own sums
};

// Memory of the grid barrier and sums (rp_handle::rsync), cleared before each
// solve: the arrival counter, its base of the next launch, the set of accumulators
// that is next and the units of the sums; three sets of 4 words for each of four sums.
constexpr int kRsCount = 0, kRsBase = 32, kRsSet = 33, kRsUnit = 34, kRsWords = 64, kRsSetWords = 16;
constexpr int kRsSync = kRsWords + 3 * 2 * kRsSetWords;
__device__ __forceinline__ void rs_reset(unsigned int* sync) {
  for (int k = threadIdx.x; k < kRsSync; k += blockDim.x)
    sync[k] = k >= kRsUnit && k < kRsWords ? (unsigned int)kFixNoUnit : 0u;
}
__device__ __forceinline__ unsigned long long* rs_words(unsigned int* sync, int set, int sum) {
  return reinterpret_cast<unsigned long long*>(sync + kRsWords) + set * kRsSetWords + sum * 4;
}

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

// Warp 0 of every block: the block's sums published, the grid met, all blocks'
// sums added in block order (so all blocks hold the same totals).
template <int NV>
__device__ __forceinline__ bool grid_total(RsFlags& sh, RsBarrier& bar, double* partials, int lane, int nw,
                                           double (&tot)[NV]) {
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
  return ok != 0;
}
template <int NV, typename T>
__device__ __forceinline__ void warp_sums(const T (&v)[NV], RsFlags& sh, int lane, int w) {
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const double s = warp_sum(v[i]);
    if (lane == 0) sh.warp[i][w] = s;
  }
}

// Grid sum of NV values a thread. Warp 0 of every block receives the totals in
// tot[] (all lanes) and calls fin(tot); then the block goes on together.
// For sums that change little from one iteration to the next: unit[i],
// kept over the iterations, is 2^-79 to 2^-80 of the last total. The threads' values
// become integers in that unit (fix_digits), the warps and the block add
// integers, and the block adds its sum, rounded to 2^-65 of the last total, to two
// 64-bit words in L2: 40 low bits with the count of values out of range above
// them, 48 high bits, and the count of arrivals in the top byte of both. A word
// whose count is complete needs no fence and no second read: one exchange instead
// of a release, an arrival, its poll, and 152 loads and their sum. Rounding: at most
// 155,648 halves (152 blocks of 1024 threads) of 2^-79 and 152 halves of 2^-65 of the
// last total, together below 2^-58; the sum is taken
// again the long way where a value reaches 2^9 of the last total, a block 2^20, or
// the total falls below 2^-7 of it (and the first time): all blocks see the same
// words and decide alike.
// (32^3: 7.1k cycles a sum the long way, 600 and 740 of them the two warp sums, 2600
// the meeting, 1800 the loads and their sum, 770 the division.)
// FENCE: the block's earlier writes are released, the others' acquired.
template <int NV, bool FENCE, typename T, typename Fin>
__device__ __forceinline__ void grid_sum_unit(const T (&v)[NV], int* unit, unsigned long long* words, RsFlags& sh,
                                              RsBarrier& bar, double* partials, int lane, int w, int nw, Fin&& fin) {
  bool quick = gridDim.x < 256;
#pragma unroll
  for (int i = 0; i < NV; ++i) quick = quick && unit[i] != kFixNoUnit;
  if (quick) {
    bool over = false;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      uint32_t u[kFixDigits];
      over = !fix_digits(v[i], unit[i], u) || over;
#pragma unroll
      for (int k = 0; k < kFixDigits; ++k) {
        u[k] = __reduce_add_sync(0xffffffffu, u[k]);
        if (lane == 0) sh.digit[i][k][w] = u[k];
      }
    }
    if (__any_sync(0xffffffffu, over) && lane == 0) sh.over = 1;
    __syncthreads();
    if (w == 0) {
      unsigned long long word = 0ull;
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        uint32_t t[kFixDigits];
#pragma unroll
        for (int k = 0; k < kFixDigits; ++k)
          t[k] = __reduce_add_sync(0xffffffffu, lane < nw ? sh.digit[i][k][lane] : 0u);
        const unsigned long long a = (unsigned long long)t[0] + ((unsigned long long)t[1] << 20);
        const long long b = (long long)t[2] + ((long long)t[3] << 20) + (long long)((unsigned long long)(long long)(int)t[4] << 40) +
                            (long long)(a >> 40);  // the sum is b 2^40 + the 40 low bits of a
        unsigned long long lo = (((a & 0xffffffffffull) + 0x2000u) >> 14) + ((unsigned long long)(b & 0x3fff) << 26);
        long long hi = b >> 14;
        const bool out = sh.over || hi >= (1ll << 46) || hi < -(1ll << 46);
        if (out) {
          lo = 1ull << 48;
          hi = 0;
        }
        if (lane == 2 * i) word = lo + (1ull << 56);
        if (lane == 2 * i + 1) word = (unsigned long long)(hi + (1ll << 47)) + (1ull << 56);
      }
      if (FENCE) __threadfence();
      if (lane < 2 * NV) asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(words + lane), "l"(word) : "memory");
      bool met = false;
      for (int64_t k = 0; k < bar.spin && !met; ++k) {
        if (lane < 2 * NV) {
          if (FENCE) asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(word) : "l"(words + lane) : "memory");
          else asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(word) : "l"(words + lane) : "memory");
        }
        met = __all_sync(0xffffffffu, lane >= 2 * NV || (word >> 56) == gridDim.x);
      }
      bool good = true;
      double tot[NV];
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const unsigned long long w0 = __shfl_sync(0xffffffffu, word, 2 * i), w1 = __shfl_sync(0xffffffffu, word, 2 * i + 1);
        const long long hi = (long long)(w1 & 0xffffffffffffffull) - ((long long)gridDim.x << 47);
        const unsigned long long lo = w0 & 0xffffffffffffull, l = ((unsigned long long)hi << 40) + lo;
        tot[i] = fix_value128((hi >> 24) + (l < lo ? 1 : 0), l, unit[i] + 14);
        good = good && ((w0 >> 48) & 255u) == 0u && fix_unit(tot[i]) >= unit[i] - 7;
      }
      __syncwarp();
      if (lane == 0) {
        sh.over = 0;
        sh.again = met && !good;
        if (!met) sh.bad = 1;
      }
      if (met && good) {
        if (lane == 0)
#pragma unroll
          for (int i = 0; i < NV; ++i) unit[i] = fix_unit(tot[i]);
        fin(tot);
      }
    }
    __syncthreads();
    if (!sh.again) return;
  }
  warp_sums(v, sh, lane, w);
  __syncthreads();
  if (w == 0) {
    double tot[NV];
    const bool ok = grid_total<NV>(sh, bar, partials, lane, nw, tot);
    if (lane == 0) {
      if (!ok) sh.bad = 1;
#pragma unroll
      for (int i = 0; i < NV; ++i)
        unit[i] = tot[i] != 0.0 && isfinite(tot[i]) ? fix_unit(tot[i]) : kFixNoUnit;
    }
    fin(tot);
  }
  __syncthreads();
}

// a / b in T without the FP64 pipe (finite a, b > 0; else as the division)
template <typename T>
__device__ __forceinline__ T ratio(double a, double b) {
  if constexpr (sizeof(T) == 8) return quot_rn(a, b);
  else return f32_rn(quot_rn(a, b));
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

// Where a product takes its vector from: its value at a global row; at(i): the
// vector seen from row i.
// The vector itself:
template <typename T>
struct RsGlobal {
  const T* x;
  __device__ __forceinline__ T operator()(int g) const { return x[g]; }
  __device__ __forceinline__ RsGlobal at(int i) const { return RsGlobal{x + i}; }
};
// z + beta p, before that sum is anywhere:
template <typename T>
struct RsFold {
  const T* z;
  const T* p;
  T beta;
  __device__ __forceinline__ T operator()(int g) const { return fma(beta, p[g], z[g]); }
  __device__ __forceinline__ RsFold at(int i) const { return RsFold{z + i, p + i, beta}; }
};

// The products of a row of the uniform layout in entry order: x seen from the row, L
// entries, their values val(e), index word wd, table entry tv of D (D and ck: what the
// checked build tests).
// (Taking the block's own rows from shared memory instead, under a predicate a lane,
// lost 4 to 20%: the products are bound by their instructions, and rank boundaries
// leave a far column in nearly every slice.)
template <typename T, class G, class Val>
__device__ __forceinline__ T rs_products(const G& x, bool valid, uint32_t wd, int32_t tv, int L, int D, const SliceCk& ck,
                                         Val&& val) {
  T g[8], s = T(0);
  if (L == 7 && __all_sync(0xffffffffu, valid)) {  // most slices: without a test an entry
#pragma unroll
    for (int e = 0; e < 7; ++e) {
      const int off = slice_offset<kIdx4>(wd, e, tv, nullptr, 0);
      g[e] = slice_ok<kIdx4>(wd, e, off, D, ck) ? x(off) : T(0);
    }
#pragma unroll
    for (int e = 0; e < 7; ++e) s = fma(val(e), g[e], s);
    return s;
  }
#pragma unroll
  for (int e = 0; e < 8; ++e)
    if (e < L) {
      const int off = slice_offset<kIdx4>(wd, e, tv, nullptr, 0);
      g[e] = valid && slice_ok<kIdx4>(wd, e, off, D, ck) ? x(off) : T(0);
    }
#pragma unroll
  for (int e = 0; e < 8; ++e)
    if (e < L) s = fma(val(e), g[e], s);
  return s;
}

// A slice of the uniform layout (4-bit indices, 1 to 8 entries a row) held
// in registers: loaded one slice ahead, across the grid barriers too, so that
// only the gathers of p wait on memory.
template <typename T>
struct RsSlice {
  T v[8];
  uint32_t wd;
  int32_t tv;
  int L;
  __device__ __forceinline__ void load(const Sliced<T>& sl, uint32_t x0, int len, uint32_t y0, uint32_t tab, int lane) {
    L = len;
    const T* p = sl.vals + x0 + lane;
    wd = ldg_stream(reinterpret_cast<const uint32_t*>(sl.ibuf) + y0 + lane);
    tv = __ldg(sl.tabs + tab + (lane & 15));
    if (L == 7) {  // a cell and its six neighbours: most slices, without a test an entry
#pragma unroll
      for (int k = 0; k < 7; ++k) v[k] = ldg_stream(p + 32 * k);
    } else {
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (k < L) v[k] = ldg_stream(p + 32 * k);
    }
  }
};

// W values of one type, moved as one access of up to 16 bytes
template <typename T, int W>
struct alignas(W * sizeof(T)) RsPack {
  T e[W];
};
template <int W, typename T>
__device__ __forceinline__ RsPack<T, W> ld_pack(const T* p) {
  return *reinterpret_cast<const RsPack<T, W>*>(p);
}
template <int W, typename T>
__device__ __forceinline__ void st_pack(T* p, const RsPack<T, W>& v) {
  *reinterpret_cast<RsPack<T, W>*>(p) = v;
}
// the same for the first m of them (global vectors: at the end of the rows, or of
// a part whose rows do not start at a multiple of W); the others read as 0
template <int W, bool RO, typename T>
__device__ __forceinline__ RsPack<T, W> ld_rows(const T* p, int m, bool whole) {
  RsPack<T, W> v;
  if (whole) {
    if constexpr (W * sizeof(T) == 16 && RO) {
      const auto q = __ldg(reinterpret_cast<const typename Vec<T>::type*>(p));
      for_each_comp<W>([&](auto c) { v.e[decltype(c)::value] = comp<decltype(c)::value>(const_cast<typename Vec<T>::type&>(q)); });
    } else {
      v = ld_pack<W>(p);
    }
    return v;
  }
#pragma unroll
  for (int e = 0; e < W; ++e) v.e[e] = e < m ? (RO ? __ldg(p + e) : p[e]) : T(0);
  return v;
}
template <int W, typename T>
__device__ __forceinline__ void st_rows(T* p, const RsPack<T, W>& v, int m, bool whole) {
  if (whole) {
    st_pack<W>(p, v);
    return;
  }
#pragma unroll
  for (int e = 0; e < W; ++e)
    if (e < m) p[e] = v.e[e];
}

// The block's slices and their products with a gathered vector. MAT (uniform
// layout): their values and index words stay in shared memory too.
template <typename T, int LAY, bool MAT = false>
struct RsMatrix {
  static constexpr bool MP = LAY == kRsParts || LAY == kRsPartsU4, U4 = LAY == kRsU4 || LAY == kRsPartsU4;
  static_assert(!MAT || U4, "only the uniform layout is kept");
  const Sliced<T>& sl;
  const Parts<T>& parts;
  const int32_t* row_ptr;
  const int32_t* col;
  const T* vals;
  int n, s0, cnt, lane, w, nw;
  int2* srow;       // MP
  uint2* sdesc;     // [cnt + 1], not U4
  uint32_t* sx;     // [cnt + 1], U4: slice s has its index words at 32 s
  uint32_t* sinfo;
  int32_t* snl;     // MP: first non-local entry of the slice's part
  const T* mv;      // MAT
  const uint32_t* mw;
  RsSlice<T> f;     // U4, not MAT: the slice fetched ahead
  NlRange fnl;

  // bytes of the records of `per` slices of at most `width` entries a row
  static int64_t tail_bytes(int lay, int64_t per, bool mat, int width) {
    const bool mp = lay == kRsParts || lay == kRsPartsU4, u4 = lay == kRsU4 || lay == kRsPartsU4;
    return (lay == kRsCsr ? 0 : (per + 1) * (u4 ? 4 : 8) + per * 4 + (mp ? per * 12 : 0)) +
           (mat ? per * kSliceRows * ((int64_t)width * (int64_t)sizeof(T) + 4) : 0);
  }
  __device__ __forceinline__ RsMatrix(const Sliced<T>& sl_, const Parts<T>& parts_, const int32_t* rp, const int32_t* c,
                                      const T* v, int n_, unsigned char* tail, int per, int width)
      : sl(sl_), parts(parts_), row_ptr(rp), col(c), vals(v), n(n_), fnl{0, 0} {
    lane = threadIdx.x & 31;
    w = threadIdx.x >> 5;
    nw = blockDim.x >> 5;
    const int S = LAY == kRsCsr ? (n + 31) / 32 : (int)sl.n_slices;
    s0 = (int)((int64_t)S * blockIdx.x / gridDim.x);
    cnt = (int)((int64_t)S * (blockIdx.x + 1) / gridDim.x) - s0;
    if (MAT) {
      T* m = reinterpret_cast<T*>(tail);
      mv = m;
      mw = reinterpret_cast<const uint32_t*>(m + (size_t)per * kSliceRows * width);
      tail += (size_t)per * kSliceRows * (width * sizeof(T) + 4);
    }
    srow = reinterpret_cast<int2*>(tail);
    sdesc = reinterpret_cast<uint2*>(srow + (MP ? per : 0));
    sx = reinterpret_cast<uint32_t*>(sdesc);
    sinfo = U4 ? sx + per + 1 : reinterpret_cast<uint32_t*>(sdesc + per + 1);
    snl = reinterpret_cast<int32_t*>(sinfo + per);
    if (LAY != kRsCsr) {
      for (int j = threadIdx.x; j <= cnt; j += blockDim.x) {
        if (U4) sx[j] = sl.desc[s0 + j].x;
        else sdesc[j] = sl.desc[s0 + j];
      }
      for (int j = threadIdx.x; j < cnt; j += blockDim.x) {
        sinfo[j] = U4 ? sl.tinfo[s0 + j] & ~kSliceW4 : sl.tinfo[s0 + j];
        if (MP) {
          const int2 r = sl.srow[s0 + j];
          srow[j] = r;
          snl[j] = (int32_t)parts.nl_off[r.y >> 6];
        }
      }
    }
    __syncthreads();
    if constexpr (MAT) {
      const uint32_t x0 = sx[0], m = sx[cnt] - x0;
      T* q = const_cast<T*>(mv);
      for (uint32_t e = threadIdx.x; e < m; e += blockDim.x)
        if (RP_IN(x0 + e, 0, sl.n_entries, kChkSliceCopy) && RP_IN(e, 0, per * kSliceRows * width, kChkSliceCopy))
          q[e] = ldg_stream(sl.vals + x0 + e);
      uint32_t* iw = const_cast<uint32_t*>(mw);
      for (int e = threadIdx.x; e < cnt * kSliceRows; e += blockDim.x)
        if (RP_IN(kSliceRows * s0 + e, 0, sl.ibuf_len, kChkSliceCopy))
          iw[e] = ldg_stream(reinterpret_cast<const uint32_t*>(sl.ibuf) + (size_t)kSliceRows * s0 + e);
      __syncthreads();
    } else if (U4 && w < cnt) {
      fetch(w);
    }
  }
  // row of slice j for this lane, or -1
  __device__ __forceinline__ int row_of(int j) const {
    if (MP) {
      const int2 r = srow[j];
      return lane < (r.y & 63) ? r.x + lane : -1;
    }
    const int i = (s0 + j) * kSliceRows + lane;
    return i < n ? i : -1;
  }
  // The block's rows in groups of W, for the passes over vectors: f(k, i, m, whole)
  // with the group's place k in shared memory, its first row i, its m rows (1 .. W)
  // and whether rows i .. i + W - 1 can be moved as one aligned access. Rows past the
  // end are zeros in shared memory.
  template <int W, typename F>
  __device__ __forceinline__ void groups(F&& f) const {
    for (int k = threadIdx.x * W; k < cnt * kSliceRows; k += blockDim.x * W) {
      int i, m;
      if (MP) {
        const int2 r = srow[k >> 5];
        i = r.x + (k & 31);
        m = min(W, (r.y & 63) - (k & 31));
      } else {
        i = s0 * kSliceRows + k;
        m = min(W, n - i);
      }
      if (m > 0) f(k, i, m, W == 1 || (!MP && m == W));
    }
  }
  // entries a row of slice j of the uniform layout (checked build: 0 where its
  // descriptor, index words or table reference leave their arrays)
  __device__ __forceinline__ int slice_len(int j) const {
    const uint32_t x0 = sx[j], x1 = sx[j + 1];
#ifdef RP_CHECK
    if (!RP_IN(x1, x0, sl.n_entries + 1, kChkSliceDesc) || !RP_IN(x1 - x0, kSliceRows, 8 * kSliceRows + 1, kChkSliceDesc) ||
        !RP_IN((int64_t)kSliceRows * (s0 + j + 1), 0, sl.ibuf_len + 1, kChkSliceDesc) ||
        !RP_IN(sinfo[j], 1, sl.tabs_len - 32 + 1, kChkSliceDesc))
      return 0;
#endif
    return (int)((x1 - x0) >> 5);
  }
  // length of its table (checked build)
  __device__ __forceinline__ int table_len(int j, int L) const {
#ifdef RP_CHECK
    return L > 0 ? __ldg(sl.tabs + sinfo[j] - 1) : 0;
#else
    (void)j, (void)L;
    return 0;
#endif
  }
  __device__ __forceinline__ NlRange nl_range(int j) const {
    const int i = row_of(j);
    return i >= 0 ? nonlocal_range<T>(parts, srow[j].y >> 6, i) : NlRange{0, 0};
  }
  __device__ __forceinline__ void fetch(int j) {
    f.load(sl, sx[j], slice_len(j), (uint32_t)(kSliceRows * (s0 + j)), sinfo[j], lane);
    if (MP) fnl = nl_range(j);
  }
  // slice j's product with x; i: row_of(j)
  template <class G>
  __device__ __forceinline__ T product(int j, int i, const G& x) {
    const bool valid = i >= 0;
    T sum = T(0);
    if constexpr (U4) {
      const G xr = x.at(valid ? i : 0);
      const int part_id = MP ? srow[j].y >> 6 : 0;
      const SliceCk ck = slice_ck<T, MP>(sl, parts, part_id, valid ? i : 0, n);
      NlRange nl{0, 0};
      if (MP) nl = MAT ? nl_range(j) : fnl;
      if constexpr (MAT) {
        const int L = slice_len(j);
        const T* v = mv + (sx[j] - sx[0]) + lane;
        const int32_t tv = __ldg(sl.tabs + sinfo[j] + (lane & 15));
        sum = rs_products<T>(xr, valid, mw[j * kSliceRows + lane], tv, L, table_len(j, L), ck,
                             [&](int e) { return v[kSliceRows * e]; });
      } else {
        const RsSlice<T> cur = f;
        fetch(j + nw < cnt ? j + nw : w);  // the last one fetches the first of the next product
        sum = rs_products<T>(xr, valid, cur.wd, cur.tv, cur.L, table_len(j, cur.L), ck, [&](int e) { return cur.v[e]; });
      }
      if (MP && nl.j0 < nl.j1) {
        const int nlo = snl[j];
        const int64_t nco = __ldg(parts.nlcol_off + part_id);
        for (int e = nl.j0; e < nl.j1; ++e) {
          const int g = nl_row_of<T>(parts, part_id, nlo, nco, e);
          if (RP_IDX_OK(g)) sum = fma(__ldg(parts.nl_vals + nlo + e), x(g), sum);
        }
      }
    } else if constexpr (LAY == kRsCsr) {
      if (valid) sum = row_dot_any<T, true>(parts, row_ptr, col, vals, x.x, i, n);
    } else {
      const int part_id = MP ? srow[j].y >> 6 : 0;
      NlRange nl{0, 0};
      if constexpr (MP)
        if (valid) nl = nonlocal_range<T>(parts, part_id, i);
      const SliceCk ck = slice_ck<T, MP>(sl, parts, part_id, i, n);
      const uint2 d0 = sdesc[j], d1 = sdesc[j + 1];
      sum = slice_sum<T, true>(d0, d1, sinfo[j], sl.vals + d0.x + lane,
                               reinterpret_cast<const uint32_t*>(sl.ibuf) + d0.y + lane, sl.tabs, x.x + (valid ? i : 0),
                               valid, lane, ck);
      if constexpr (MP)
        if (valid) sum = nonlocal_sum<T, true>(parts, part_id, nl, x.x, sum);
    }
    return sum;
  }
};

// The launch of a resident kernel, in one of its forms (the first that fits): how
// many vectors it keeps in shared memory, whether the matrix too, and at most how
// many rows a block.
struct ResidentPlan {
  void* fn = nullptr;  // nullptr: the streaming kernels run
  int grid = 0, threads = 0, smem = 0, rows = 0, width = 0;
  int32_t form = RP_FORM_STREAMING;
};
struct ResidentForm {
  int vecs;
  bool mat;
  int max_rows;
  int id;
  int32_t form = RP_FORM_RESIDENT;
};
// Limits below this keep to the streaming kernels. A poll of the arrival counter is
// an L2 round trip (0.4 us), a block waits for the slowest one's pass of up to 0.1
// ms; a caller's small limit was chosen for the mbarrier probes of the streaming
// products, or for kernels without any wait (CSR), which it suffices for.
constexpr int64_t kResidentSpin = int64_t(1) << 16;
inline int64_t resident_spin(const rp_handle* h) {
#ifdef RP_CHECK
  if (h->check_spin >= 0) return h->check_spin;
#endif
  return h->opts.spin_limit;
}
// A cooperative launch can be refused (in a graph under MPS, for instance): the
// caller takes the streaming kernels then.
inline cudaError_t cooperative_node(const rp_handle* h, cudaGraphNode_t node) {
#ifdef RP_CHECK
  if (h->check_refuse) return cudaErrorNotSupported;
#else
  (void)h;
#endif
  cudaLaunchAttributeValue coop{};
  coop.cooperative = 1;
  return cudaGraphKernelNodeSetAttribute(node, cudaLaunchAttributeCooperative, &coop);
}
inline cudaError_t launch_resident(const rp_handle* h, const ResidentPlan& p, void* argp, cudaStream_t s) {
#ifdef RP_CHECK
  if (h->check_refuse) return cudaErrorNotSupported;
#else
  (void)h;
#endif
  void* args[1] = {argp};
  return cudaLaunchCooperativeKernel(p.fn, dim3((unsigned)p.grid), dim3((unsigned)p.threads), args, (size_t)p.smem, s);
}
// How large a system in another layout than the uniform one may be. The streaming
// products hide the latency of its loads behind twice the warps, so the resident
// form loses where those loads miss. (us an iteration there, then here; 5 to 20
// entries a row.)
//
// Sliced, FP32: at most `l2` bytes of values, indices and tables; beyond, they miss L2
// (PCG: 76 MB 72.0, 53.8 and 69.2, 56.2; 81 MB 75.3, 75.0; 100 MB 95.5, 122.2; 131 MB
// 114, 141; BiCGStab: 74 MB 162, 98; 76 MB 147, 161 and 159, 152; 81 MB 167, 172). FP64
// stays ahead (480 MB: 479, 459), save with r and q alone on chip and tables that slices
// do not share (a mesh numbered at random, 33 MB of them: 131, 140).
//
// CSR: threads read their rows piece by piece, and shared memory has to leave L1 a part
// of what the rows of all threads take, here per form and for several parts.
//   FP64, four vectors: 0.22 152, 341; 0.48 79, 83; 0.72 100, 77; 0.80 57, 48; parts 0.81
//     64, 69; 1.19 55, 44 (BiCGStab 0.48 155, 171; 0.80 115, 104; parts 0.81 126, 147)
//   FP64, two: 0.50 218, 260; 0.96 88, 102; 1.09 108, 93; parts 1.25 90, 97; 1.53 81, 80
//   FP32: 0.28 178, 426; 0.72 56.6, 59.8; 0.85 122, 109; 1.03 54.6, 55.5 (BiCGStab 119,
//     108); parts 1.24 60, 81; 1.61 57.0, 57.7; 1.97 52, 47
constexpr int64_t kOwnTables = 16 * 1024 * 1024;  // more bytes of tables: slices do not share them
constexpr int64_t kL1Bytes = 256 * 1024;          // L1 and shared memory of an SM
constexpr double csr_share(bool fp64, int vecs, bool parts) {
  if (parts) return fp64 && vecs == 4 ? 0.9 : 1.5;
  return !fp64 ? 0.8 : vecs == 4 ? 0.6 : 1.0;
}

// fn_of(layout, form): the instance, or nullptr where there is none
template <typename T, typename Fn>
ResidentPlan plan_resident(const rp_handle* h, const Sliced<T>& sl, int64_t n, int64_t l2,
                           std::initializer_list<ResidentForm> forms, Fn&& fn_of) {
  ResidentPlan p;
  int coop = 0, smem_max = 0;
  if (n == 0 || h->opts.spin_limit < kResidentSpin) return p;
  if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, h->device) != cudaSuccess || !coop ||
      cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, h->device) != cudaSuccess) {
    cudaGetLastError();
    return p;
  }
  const bool u4 = sl.u4 != 0;
  const int lay = sl.n_slices == 0 ? kRsCsr : sl.srow ? (u4 ? kRsPartsU4 : kRsParts) : u4 ? kRsU4 : kRsSliced;
  const int64_t S = lay == kRsCsr ? (n + 31) / 32 : sl.n_slices;
  const int grid = (int)std::min<int64_t>(h->num_sms, S);
  const int64_t per = (S + grid - 1) / grid;  // slices a block at most
  const bool general = lay == kRsSliced || lay == kRsParts;
  const int64_t tables = 4 * sl.tabs_len;
  if (general && sizeof(T) == 4 && 4 * sl.n_entries + 4 * sl.ibuf_len + tables > l2) return p;
  const double row_bytes = (double)(h->nnz + h->nl_nnz) * (sizeof(T) + 4.0) / (double)n;
  for (const ResidentForm& f : forms) {
    if ((f.mat && !u4) || per * 32 > f.max_rows || (general && f.vecs < 4 && tables > kOwnTables)) continue;
    void* fn = fn_of(lay, f);
    if (!fn) continue;
    const int64_t need =
        per * 32 * f.vecs * (int64_t)sizeof(T) + RsMatrix<T, kRsCsr>::tail_bytes(lay, per, f.mat, h->sl_width);
    const int threads = 32 * (int)std::min<int64_t>(std::max<int64_t>(per, 4), (f.mat ? kRsThreads<T, true> : kRsThreads<T, false>) / 32);
    if (lay == kRsCsr &&
        (double)(kL1Bytes - need) < csr_share(sizeof(T) == 8, f.vecs, h->n_parts > 1) * threads * row_bytes)
      continue;
    cudaFuncAttributes at;
    int nb = 0;
    // the kernel's own (static) shared memory comes off the block's limit
    if (cudaFuncGetAttributes(&at, fn) == cudaSuccess && need <= smem_max - (int)at.sharedSizeBytes &&
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max - (int)at.sharedSizeBytes) ==
            cudaSuccess &&
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, threads, (size_t)need) == cudaSuccess && nb >= 1)
      return ResidentPlan{fn, grid, threads, (int)need, (int)(per * 32), h->sl_width, f.form};
    cudaGetLastError();
  }
  return p;
}

}  // namespace rp
