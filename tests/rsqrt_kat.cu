// rsqrt_householder (the pivots' reciprocal square root, csrc/fifa_level.cuh) and the
// library's rsqrt on n doubles in host memory; a cudaError_t.
#include "fifa_level.cuh"

__global__ void k_rsqrt(const double* __restrict__ x, double* __restrict__ mine, double* __restrict__ lib, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  mine[i] = rsqrt_householder(x[i]);
  lib[i] = rsqrt(x[i]);
}

extern "C" int rsqrt_kat(const double* x, double* mine, double* lib, int n) {
  double* d = nullptr;
  const size_t b = sizeof(double) * n;
  cudaError_t e = cudaMalloc((void**)&d, 3 * b);
  if (e != cudaSuccess) return e;
  e = cudaMemcpy(d, x, b, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    k_rsqrt<<<(n + 255) / 256, 256>>>(d, d + n, d + 2 * n, n);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(mine, d + n, b, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(lib, d + 2 * n, b, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e;
}
