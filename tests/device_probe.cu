// The library's internal device functions, called one by one: compiled by the
// tests (device_probe.py) from the library's own headers.
#include "rp_resident.cuh"

namespace {

__global__ void k_quotients(const double* a, const double* b, double* out, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = rp::quot_rn(a[i], b[i]);
}

// One sum of two values a thread by a grid of blocks, in units taken from `last` (0: none
// yet), and then a second one of the same values: totals and units left by block 0,
// out[4 b ..] what block b holds after each; bad[b]: a wait ran out.
__global__ void __launch_bounds__(1024, 1)
    k_grid_sums(const double* v, const double* last, unsigned int* sync, int64_t spin, double* partials, double* out,
                int* bad) {
  __shared__ rp::RsFlags sh;
  __shared__ int unit[2];
  if (threadIdx.x == 0) {
    sh.stop = sh.bad = sh.over = sh.again = 0;
    for (int i = 0; i < 2; ++i) unit[i] = last[i] == 0.0 ? rp::kFixNoUnit : rp::fix_unit(last[i]);
  }
  __syncthreads();
  rp::RsBarrier bar{sync, 0u, spin};
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int64_t at = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, all = (int64_t)gridDim.x * blockDim.x;
  const double x[2] = {v[at], v[all + at]};
  for (int k = 0; k < 2 && !sh.bad; ++k)
    rp::grid_sum_unit<2, true>(x, unit, rp::rs_words(sync, k, 0), sh, bar, partials + 2 * k * gridDim.x, lane, w, nw,
                               [&](const double (&tot)[2]) {
                                 if (lane < 2) out[4 * blockIdx.x + 2 * k + lane] = tot[lane];
                               });
  if (threadIdx.x == 0) bad[blockIdx.x] = sh.bad;
}
__global__ void k_sync_reset(unsigned int* sync) { rp::rs_reset(sync); }

}  // namespace

// blocks <= the SMs; v: two rows of blocks x threads; out: 4 a block; bad: 1 a block
extern "C" int probe_grid_sums(const double* v, const double* last, int blocks, int threads, int64_t spin, double* out,
                               int* bad, void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
  unsigned int* sync;
  double* partials;
  if (cudaMalloc(&sync, sizeof(unsigned int) * rp::kRsSync) != cudaSuccess) return (int)cudaGetLastError();
  if (cudaMalloc(&partials, sizeof(double) * 4 * blocks) != cudaSuccess) return (int)cudaGetLastError();
  k_sync_reset<<<1, rp::kRsSync, 0, s>>>(sync);
  void* args[] = {&v, &last, &sync, &spin, &partials, &out, &bad};
  cudaLaunchCooperativeKernel((void*)k_grid_sums, dim3(blocks), dim3(threads), args, 0, s);
  const int e = (int)cudaStreamSynchronize(s);
  cudaFree(sync);
  cudaFree(partials);
  return e;
}

extern "C" int probe_inner_runs(int stop, int status) { return rp::inner_runs(stop, status) ? 1 : 0; }

extern "C" int probe_quotients(const double* a, const double* b, double* out, int64_t n, void* stream) {
  k_quotients<<<1024, 256, 0, (cudaStream_t)stream>>>(a, b, out, n);
  return (int)cudaGetLastError();
}
