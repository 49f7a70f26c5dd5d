// Test-only probe: the library's own elementary functions (device_math.cuh), value by value.
#include "device_math.cuh"

__global__ void exp_kernel(const double* x, double* y, int n) {
  __shared__ unsigned long long pow2[rewl::kPow2];
  if (threadIdx.x < rewl::kPow2) pow2[threadIdx.x] = rewl::pow2_entry(threadIdx.x);
  __syncthreads();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) y[i] = rewl::exp_fixed(x[i], pow2);
}

__global__ void reciprocal_kernel(const float* x, float* y, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) y[i] = rewl::reciprocal(x[i]);
}

template <class T, class F>
static int apply(const T* x, T* y, int n, F launch) {
  T *dx = nullptr, *dy = nullptr;
  cudaError_t e = cudaMalloc(&dx, sizeof(T) * (size_t)n);
  if (e == cudaSuccess) e = cudaMalloc(&dy, sizeof(T) * (size_t)n);
  if (e == cudaSuccess) e = cudaMemcpy(dx, x, sizeof(T) * (size_t)n, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    launch(dx, dy);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(y, dy, sizeof(T) * (size_t)n, cudaMemcpyDeviceToHost);
  cudaFree(dx);
  cudaFree(dy);
  return (int)e;
}

extern "C" int probe_exp(const double* x, double* y, int n) {
  return apply(x, y, n, [n](const double* a, double* b) { exp_kernel<<<256, 256>>>(a, b, n); });
}
extern "C" int probe_reciprocal(const float* x, float* y, int n) {
  return apply(x, y, n, [n](const float* a, float* b) { reciprocal_kernel<<<256, 256>>>(a, b, n); });
}
