// The library's internal device functions, called one by one: compiled by the
// tests (device_probe.py) from the library's own headers.
#include "rp_values.cuh"

namespace {

__global__ void k_quotients(const double* a, const double* b, double* out, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = rp::quot_rn(a[i], b[i]);
}

}  // namespace

extern "C" int probe_inner_runs(int stop, int status) { return rp::inner_runs(stop, status) ? 1 : 0; }

extern "C" int probe_quotients(const double* a, const double* b, double* out, int64_t n, void* stream) {
  k_quotients<<<1024, 256, 0, (cudaStream_t)stream>>>(a, b, out, n);
  return (int)cudaGetLastError();
}
