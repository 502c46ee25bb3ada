// The prompt GEMM's silu over an array, for test_gpu_silu.py.
#include "ada_gemm_pair.cuh"

__global__ void k_silu(const float *x, float *y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = ada::silu(x[i]);
}

extern "C" int silu_run(const float *x, float *y, int n) {
  k_silu<<<(n + 255) / 256, 256>>>(x, y, n);
  return cudaDeviceSynchronize() == cudaSuccess ? 0 : 1;
}
