// The reciprocal square root and square root of the Cholesky pivots (csrc/rsqrt.h) beside CUDA's rsqrt and sqrt, for their
// test.  Not part of the library's C ABI.
#include "../csrc/rsqrt.h"

namespace {
__global__ void k_rsqrt(int n, const double *d, double *out) {   // out[4][n]
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double r = librpa::fast_rsqrt(d[i]);
  out[i] = r;
  out[n + i] = librpa::sqrt_from(d[i], r);
  out[2 * n + i] = rsqrt(d[i]);
  out[3 * n + i] = sqrt(d[i]);
}
}  // namespace

// host arrays d[n], out[4][n]; returns a cudaError_t
extern "C" int librpa_probe_rsqrt(int n, const double *d, double *out) {
  double *p = nullptr;
  cudaError_t e = cudaMalloc(&p, 5 * (size_t)n * sizeof(double));
  if (e != cudaSuccess) return (int)e;
  e = cudaMemcpy(p, d, (size_t)n * sizeof(double), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    k_rsqrt<<<(n + 255) / 256, 256>>>(n, p, p + n);
    e = cudaMemcpy(out, p + n, 4 * (size_t)n * sizeof(double), cudaMemcpyDeviceToHost);
  }
  cudaFree(p);
  return (int)e;
}
