// Test helper: T -= Z Z^T (lower triangle) by the library's tensor-core tiles
// (kkt_oz.cuh), one CTA, operands in device memory. Built by the tests with
// nvcc; not part of the library.
#include <cuda_runtime.h>

#include "../../paper_2511_00946_gb300/csrc/kkt_oz.cuh"

namespace {
namespace oz = kkt::oz;
__global__ void k_probe(double* Z, int ldz, int rows, int n, double* T, int ldt, int* f) {
  for (int r = threadIdx.x; r < rows; r += blockDim.x) {
    oz::u64* z = (oz::u64*)(Z + r * ldz);
    int em = 0;
    for (int k = 0; k < n; ++k) em = max(em, oz::mag(z[k]));
    f[r] = oz::row_exp(em);
    if (f[r] != oz::kFp64Row)
      for (int k = 0; k < n; ++k) z[k] = oz::encode(z[k], f[r]);
  }
  __syncthreads();
  int w = 0;
  for (int a = 0; a < rows; a += 16)
    for (int b = 0; b < min(a + 16, rows); b += 8, ++w)
      if (w % (int)(blockDim.x >> 5) == (int)(threadIdx.x >> 5))
        oz::tile(T, ldt, Z, f, Z, f, 0, ldz, a, rows, b, rows, n, threadIdx.x & 31);
}
}  // namespace

// Z [rows][ldz] (overwritten), T [rows][ldt], f [rows]: device arrays
extern "C" int oz_probe(double* Z, int ldz, int rows, int n, double* T, int ldt, int* f) {
  if (rows < 1 || n < 1 || ldz < n || ldt < rows) return (int)cudaErrorInvalidValue;
  k_probe<<<1, 256>>>(Z, ldz, rows, n, T, ldt, f);
  const int e = (int)cudaGetLastError();
  return e ? e : (int)cudaDeviceSynchronize();
}
