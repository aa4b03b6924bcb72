// Test shim: the library's own arithmetic (nle_device.cuh) beside CUDA's, for
// tests/test_gpu_arith.py.  Built by that test with nvcc; not part of the library.
#include "../paper_1312_1553_gb300/csrc/nle_device.cuh"

using namespace nle;

// arguments [0, 2^32) whose conversion differs: in the bits or, for a NaN, in being one
__global__ void k_wide(unsigned long long *bad) {
  const unsigned long long step = (unsigned long long)gridDim.x * blockDim.x;
  unsigned long long n = 0;
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < 1ull << 32; i += step) {
    const float f = __uint_as_float((unsigned)i);
    const double a = wide(f), b = double(f);
    n += f != f ? a == a : __double_as_longlong(a) != __double_as_longlong(b);
  }
  if (n) atomicAdd(bad, n);
}

extern "C" int shim_wide(unsigned long long *bad) {
  unsigned long long *d = nullptr;
  cudaMalloc(&d, 8), cudaMemset(d, 0, 8);
  k_wide<<<1216, 256>>>(d);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpy(bad, d, 8, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e == cudaSuccess ? 0 : 1;
}

__global__ void k_quotient(int n, const double *t, const double *d, double *q, double *div) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const double inv = 1.0 / d[i];
    q[i] = quotient(t[i], d[i], inv);
    div[i] = t[i] / d[i];
  }
}

// host arrays of n doubles
extern "C" int shim_quotient(int n, const double *t, const double *d, double *q, double *div) {
  double *dev = nullptr;
  const size_t b = (size_t)n * sizeof(double);
  if (cudaMalloc(&dev, 4 * b) != cudaSuccess) return 1;
  cudaMemcpy(dev, t, b, cudaMemcpyHostToDevice), cudaMemcpy(dev + n, d, b, cudaMemcpyHostToDevice);
  k_quotient<<<1216, 256>>>(n, dev, dev + n, dev + 2 * (size_t)n, dev + 3 * (size_t)n);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpy(q, dev + 2 * (size_t)n, b, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(div, dev + 3 * (size_t)n, b, cudaMemcpyDeviceToHost);
  cudaFree(dev);
  return e == cudaSuccess ? 0 : 1;
}
