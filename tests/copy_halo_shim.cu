// Test shim: copy_halo (nle_device.cuh) by one CTA's copying warps alone, for
// tests/test_gpu_copy_halo.py.  Built by that test with nvcc; not part of the library.
#include "../paper_1312_1553_gb300/csrc/nle_device.cuh"

using namespace nle;

extern __shared__ __align__(16) unsigned char window[];

template <typename T>
__global__ void k_copy(const int32_t *hpos, int nh, const T *x, long long spin_ns, State *st, T *out, int *arrived,
                       long long *cycles) {
  __shared__ Shared sh;
  const int m = threadIdx.x >> 5;
  if (threadIdx.x < COPY_WARPS) sh.arrived[threadIdx.x] = 32 * threadIdx.x;
  for (int i = threadIdx.x; i < nh; i += blockDim.x) reinterpret_cast<T *>(window)[i] = T(-1);
  __syncthreads();
  const long long t0 = clock64();
  copy_halo<T>(hpos, nh, m, x, smem_addr(window), sh, spin_ns, st);
  if ((threadIdx.x & 31) == 0) cycles[m] = clock64() - t0, arrived[m] = sh.arrived[m];
  __syncthreads();
  for (int i = threadIdx.x; i < nh; i += blockDim.x) out[i] = reinterpret_cast<T *>(window)[i];
}

template <typename T>
static int run(const int32_t *hpos, int nh, const T *x, int nx, long long spin_ns, T *out, int *arrived,
               long long *cycles, int *err) {
  if (nh < 1 || nh * sizeof(T) > 16384) return 1;
  int32_t *dpos = nullptr;
  T *dx = nullptr, *dout = nullptr;
  State *st = nullptr;
  int *darr = nullptr;
  long long *dcyc = nullptr;
  cudaMalloc(&dpos, nh * 4), cudaMalloc(&dx, nx * sizeof(T)), cudaMalloc(&dout, nh * sizeof(T));
  cudaMalloc(&st, sizeof(State)), cudaMalloc(&darr, 16), cudaMalloc(&dcyc, 32);
  cudaMemset(st, 0, sizeof(State));
  cudaMemcpy(dpos, hpos, nh * 4, cudaMemcpyHostToDevice);
  cudaMemcpy(dx, x, nx * sizeof(T), cudaMemcpyHostToDevice);
  k_copy<T><<<1, 32 * COPY_WARPS, nh * sizeof(T)>>>(dpos, nh, dx, spin_ns, st, dout, darr, dcyc);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  State s;
  cudaMemcpy(&s, st, sizeof s, cudaMemcpyDeviceToHost);
  cudaMemcpy(out, dout, nh * sizeof(T), cudaMemcpyDeviceToHost);
  cudaMemcpy(arrived, darr, 16, cudaMemcpyDeviceToHost);
  cudaMemcpy(cycles, dcyc, 32, cudaMemcpyDeviceToHost);
  *err = s.err;
  cudaFree(dpos), cudaFree(dx), cudaFree(dout), cudaFree(st), cudaFree(darr), cudaFree(dcyc);
  return e == cudaSuccess ? 0 : 2;
}

extern "C" int shim_copy_f32(const int32_t *hpos, int nh, const float *x, int nx, long long spin_ns,
                             float *out, int *arrived, long long *cycles, int *err) {
  return run<float>(hpos, nh, x, nx, spin_ns, out, arrived, cycles, err);
}
extern "C" int shim_copy_f64(const int32_t *hpos, int nh, const double *x, int nx, long long spin_ns,
                             double *out, int *arrived, long long *cycles, int *err) {
  return run<double>(hpos, nh, x, nx, spin_ns, out, arrived, cycles, err);
}
