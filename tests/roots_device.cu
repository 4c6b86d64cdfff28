// The FP64 roots and reciprocal of su2_device.cuh on the GPU, for
// tests/test_gpu_fixed_point.py.
#include "su2_device.cuh"

static __global__ void k_roots(const double* v, int n, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  out[i] = su2::rsqrt64(v[i]);
  out[n + i] = su2::sqrt64(v[i]);
  out[2 * n + i] = su2::half_inverse64(v[i]);
}

// v, out: host arrays of n and 3 n doubles.  Returns a CUDA error.
extern "C" int roots(const double* v, int n, double* out) {
  double *d = nullptr, *o = nullptr;
  cudaError_t e = cudaMalloc(&d, n * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&o, 3 * (size_t)n * sizeof(double));
  if (e == cudaSuccess) e = cudaMemcpy(d, v, n * sizeof(double), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) k_roots<<<(n + 255) / 256, 256>>>(d, n, o);
  if (e == cudaSuccess) e = cudaMemcpy(out, o, 3 * (size_t)n * sizeof(double), cudaMemcpyDeviceToHost);
  cudaFree(d);
  cudaFree(o);
  return (int)e;
}
