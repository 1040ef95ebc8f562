// rsqrt_fp64 and rcp_fp64 (csrc/fp64_ops.cuh) over an array; built by
// tests/test_gpu_fp64_ops.py.
#include "fp64_ops.cuh"

__global__ void k(const double* x, int n, double* r, double* q) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    r[i] = ifmm::rsqrt_fp64(x[i]);
    q[i] = ifmm::rcp_fp64(x[i]);
  }
}

extern "C" int fp64_ops(const double* x, int n, double* r, double* q) {
  double* d = nullptr;
  if (cudaMalloc((void**)&d, sizeof(double) * 3 * n) != cudaSuccess) return 1;
  cudaMemcpy(d, x, sizeof(double) * n, cudaMemcpyHostToDevice);
  k<<<(n + 255) / 256, 256>>>(d, n, d + n, d + 2 * n);
  cudaError_t e = cudaMemcpy(r, d + n, sizeof(double) * n, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(q, d + 2 * n, sizeof(double) * n, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e != cudaSuccess;
}
