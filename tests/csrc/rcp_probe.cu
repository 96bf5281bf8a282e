// Test helper: the pivot reciprocal of kkt_numerics.cuh, elementwise. Built by
// the tests with nvcc; not part of the library.
#include <cuda_runtime.h>

#include "../../paper_2511_00946_gb300/csrc/kkt_numerics.cuh"

namespace {
__global__ void k_probe(const double* in, double* out, double* ok, long long count) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  ok[i] = kkt::pivot_rcp_ok(in[i]) ? 1.0 : 0.0;
  out[i] = kkt::pivot_rcp(in[i]);
}
}  // namespace

extern "C" int rcp_probe(const double* in, double* out, double* ok, long long count) {
  if (count <= 0) return 0;
  k_probe<<<(unsigned)((count + 255) / 256), 256>>>(in, out, ok, count);
  const int e = (int)cudaGetLastError();
  return e ? e : (int)cudaDeviceSynchronize();
}
