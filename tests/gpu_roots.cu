// Test harness for the root of csrc/s2_internal.cuh (compiled by
// tests/test_gpu_roots.py; not part of the library).
#include <cuda_runtime.h>

#include "../paper_2304_05494_gb300/csrc/s2_internal.cuh"

namespace {
__global__ void k_roots(const double *in, double *out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = s2::sqrt_pos(in[i]);
}
}  // namespace

extern "C" int roots_run(const double *in, double *out, int n) {
  double *din = nullptr, *dout = nullptr;
  if (cudaMalloc(&din, n * sizeof(double)) != cudaSuccess || cudaMalloc(&dout, n * sizeof(double)) != cudaSuccess)
    return 1;
  cudaMemcpy(din, in, n * sizeof(double), cudaMemcpyHostToDevice);
  k_roots<<<(n + 255) / 256, 256>>>(din, dout, n);
  const cudaError_t e = cudaMemcpy(out, dout, n * sizeof(double), cudaMemcpyDeviceToHost);
  cudaFree(din);
  cudaFree(dout);
  return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? 0 : 2;
}
