// Test harness for the power law and logarithm of csrc/s2_power.cuh
// (compiled by tests/test_gpu_power.py; not part of the library).
#include <cuda_runtime.h>
#include <string.h>

#include "../paper_2304_05494_gb300/csrc/s2_power.cuh"

using namespace s2;

namespace {
__global__ void k_power(int which, const double *in, double *out, int n, Dev d) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = which == 0 ? viscosity_fixed(d, in[i]) : FixedLog{d.powt}(in[i]);
}
}  // namespace

// which = 0: in^omega (T_ref = Re = 1), 1: ln(in).
extern "C" int power_run(int which, const double *in, double *out, int n, double omega) {
  Dev d;
  memset(&d, 0, sizeof(d));
  d.inv_t_ref = d.inv_re = 1.0;
  d.visc_exp = omega;
  d.visc_exp_f = (float)omega;
  PowTab host;
  pow_setup(d, host);
  double *din = nullptr, *dout = nullptr;
  PowTab *tab = nullptr;
  if (cudaMalloc(&din, n * sizeof(double)) != cudaSuccess || cudaMalloc(&dout, n * sizeof(double)) != cudaSuccess ||
      cudaMalloc(&tab, sizeof(PowTab)) != cudaSuccess)
    return 1;
  d.powt = tab;
  cudaMemcpy(tab, &host, sizeof(PowTab), cudaMemcpyHostToDevice);
  cudaMemcpy(din, in, n * sizeof(double), cudaMemcpyHostToDevice);
  k_power<<<(n + 255) / 256, 256>>>(which, din, dout, n, d);
  const cudaError_t e = cudaMemcpy(out, dout, n * sizeof(double), cudaMemcpyDeviceToHost);
  cudaFree(din);
  cudaFree(dout);
  cudaFree(tab);
  return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? 0 : 2;
}
