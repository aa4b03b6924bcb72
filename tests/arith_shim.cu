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
