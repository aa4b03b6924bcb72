// Allocation-free application of the incomplete-Cholesky preconditioner,
// c = (L L^T)^{-1} g, for callers that must not allocate device memory.
//
// All temporary storage of this entry point lives in one file-scope device
// array (nle_noalloc_scratch): the intermediate vector z = L^{-1} g and an
// error word.  Host code never uses the array's name as an address; it asks
// the runtime for the array's device address once per device.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <mutex>
#include <string>
#include <type_traits>

#include "../../include/nle.h"
#include "nle_device.cuh"

namespace {

constexpr int64_t kMaxN = NLE_NOALLOC_MAX_N;
constexpr int kMaxDevices = 64;

// z (kMaxN doubles) followed by a small control block (error word).
static __device__ __align__(256) double nle_noalloc_scratch[kMaxN + 32];

std::mutex g_mu;
double *g_scratch[kMaxDevices] = {nullptr};

// Set z and c to the not-yet-computed marker and clear the error word.
__global__ void k_na_fill(double *z, double *c, int64_t n, int *err) {
  const double sent = nle::sentinel<double>();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    z[i] = sent;
    c[i] = sent;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *err = 0;
}

constexpr int kWarps = 32;    // warps of a CTA
constexpr int kRows = 4;      // rows a warp has open at a time, 32 / kRows lanes each
constexpr int kWide = 32;     // mean entries of a row from which a warp takes one row at a time
constexpr int kLong = 64;     // entries of a lane from which it takes four at a time
constexpr int kSleep = 40;    // ns between two rounds of looks that found nothing

// Four rows per warp, eight lanes a row and two entries of a lane in flight (one row
// and 32 lanes for factors with wide rows); groups of four rows are taken
// round-robin in order (ascending for the lower factor, descending for the
// upper one).  A row waits only for rows of earlier
// groups and for earlier rows of its own.  The warps are all resident
// (cooperative launch), and a warp looks at the missing values of all its
// rows in turn without stopping at one, so every wait ends.  Entries whose
// column is not strictly below (above) the row, or outside [0, n), are skipped
// and reported; every wait is bounded.
//
// Bound by the latency of one dependency (store, look through L2, sum) times
// the number of dependencies in a line that the rows in flight cannot overlap.
// So many rows are open at a time (32 warps an SM x 4: 19,456, nine planes of
// a 45 x 50 x 55 grid), and what does not depend on the
// solution (pointers, coefficients, right-hand side, reciprocal pivot) is read
// before the first look.  A lane adds its entries in order and eight lanes
// meet in a tree: the sum does not depend on when values arrive.
// Both solves together, against one warp per row that divided after the last
// value arrived and read its row after the row before was done (1,216 rows in
// flight): n = 123,750 7-point 28.7 -> 1.39 ms.  With 8 and 16 warps an SM
// 5.39 and 2.89 ms, with 2 rows a warp (16 lanes each) 3.28, with 8 rows 1.60
// (2.65 against 2.52 on 300 x 350 5-point, 1.91 against 2.34 on 27-point
// 40^3); no pause, 40 ns and 200 ns between looks 1.39, 1.39, 1.41.
// A long row is bound by its own reads: a look at 16 entries costs two dependent
// reads through L2, 0.65 us.  Factors with more than kWide entries a row on average give a row
// all 32 lanes (one warp per row before / 8 lanes / 32 lanes: 50,000 rows of 64 and 200 random
// entries 5.1 / 6.7 / 2.9 and 19.9 / 39.8 / 11.7 ms, a dense triangle of 1,500 18.1 / 32.3 / 9.3,
// 20,000 rows of 50 neighbours 56.5 with 8 lanes and 42.9 with 32, of 30 39.1 and 41.5); a
// lane with more than kLong entries left takes four at a time while their values are
// there (a hub of 9,000 neighbours 0.24 / 0.36 / 0.25), in a loop of its own, since the others
// lose 3 % by it.
template <bool LOWER, int ROWS>
__device__ __forceinline__ void na_rows(int64_t n, const int32_t *rp, const int32_t *col, const double *val,
                                        const double *diag, const double *rhs, double *x, int *err,
                                        long long lim_cycles) {
  constexpr unsigned kFull = 0xffffffffu;
  constexpr int kLanes = 32 / ROWS;
  const int lane = threadIdx.x & 31, sub = lane % kLanes;
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t g = w; g * ROWS < n; g += nw) {
    const int64_t it = g * ROWS + lane / kLanes;
    const int64_t r = LOWER ? it : n - 1 - it;
    bool open = it < n;  // the row has not been published
    int e = 0, e1 = 0;
    double b = 0.0, d = 1.0;
    if (open) {
      e = __ldg(rp + r) + sub;
      e1 = __ldg(rp + r + 1);
      b = __ldg(rhs + r);
      d = __ldg(diag + r);
    }
    int c[2];
    double v[2], xv[2];
    bool miss[2];
    auto fetch = [&] {
#pragma unroll
      for (int t = 0; t < 2; t++) {
        const int k = e + t * kLanes;
        c[t] = k < e1 ? __ldg(col + k) : 0;
        v[t] = k < e1 ? __ldg(val + k) : 0.0;
        xv[t] = 0.0;
        miss[t] = k < e1;
        if (miss[t] && !(LOWER ? (c[t] >= 0 && c[t] < r) : (c[t] > r && c[t] < n))) {
          atomicCAS(err, 0, (int)NLE_ERR_CSR);
          v[t] = 0.0;
          miss[t] = false;
        }
      }
    };
    fetch();
    const double inv = 1.0 / d;
    double acc = 0.0;
    auto solve = [&](auto bulk) {
      long long c0 = clock64();
      while (true) {
        if (miss[0]) xv[0] = nle::ld_relaxed(x + c[0]);
        if (miss[1]) xv[1] = nle::ld_relaxed(x + c[1]);
        miss[0] = miss[0] && nle::is_sent(xv[0]);
        miss[1] = miss[1] && nle::is_sent(xv[1]);
        bool moved = e < e1 && !miss[0] && !miss[1];
        if (moved) {
          acc += v[0] * xv[0];
          acc += v[1] * xv[1];
          e += 2 * kLanes;
          if constexpr (decltype(bulk)::value) {
            for (int q = 0; q < 8 && e1 - e > 4 * kLanes; q++) {
              int cb[4];
              double xb[4];
              bool all = true;
#pragma unroll
              for (int t = 0; t < 4; t++) cb[t] = __ldg(col + e + t * kLanes);
#pragma unroll
              for (int t = 0; t < 4; t++) {
                const bool ok = LOWER ? (cb[t] >= 0 && cb[t] < r) : (cb[t] > r && cb[t] < n);
                xb[t] = ok ? nle::ld_relaxed(x + cb[t]) : nle::sentinel<double>();
              }
#pragma unroll
              for (int t = 0; t < 4; t++) all = all && !nle::is_sent(xb[t]);
              if (!all) break;  // the two at a time wait, and report a column out of place
#pragma unroll
              for (int t = 0; t < 4; t++) acc += __ldg(val + e + t * kLanes) * xb[t];
              e += 4 * kLanes;
            }
          }
          if (e < e1) fetch();
        }
        const unsigned ready = __ballot_sync(kFull, e >= e1);
        constexpr unsigned kAll = kFull >> (32 - kLanes);
        const bool publish = open && ((ready >> (lane - sub)) & kAll) == kAll;
        if (__any_sync(kFull, publish)) {
          double s = acc;
#pragma unroll
          for (int o = kLanes / 2; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
          if (publish && sub == 0) nle::st_relaxed(x + r, nle::quotient(b - s, d, inv));
          if (publish) open = false;
          if (!__any_sync(kFull, open)) break;
          moved = true;
        }
        if (__any_sync(kFull, moved)) {
          c0 = clock64();
        } else {
          if (clock64() - c0 > lim_cycles) {
            // nothing came for this warp: report, and go on with zeros
#pragma unroll
            for (int t = 0; t < 2; t++)
              if (miss[t]) {
                atomicCAS(err, 0, (int)NLE_ERR_TIMEOUT);
                xv[t] = 0.0;
                miss[t] = false;
              }
          }
          __nanosleep(kSleep);
        }
      }
    };
    if (ROWS == 1 || __any_sync(kFull, e1 - e > kLong * kLanes)) solve(std::true_type());
    else solve(std::false_type());
  }
}

template <bool LOWER>
__global__ void __launch_bounds__(32 * kWarps) k_na_solve(int64_t n, const int32_t *rp, const int32_t *col,
                                                          const double *val, const double *diag, const double *rhs,
                                                          double *x, int *err, long long lim_cycles) {
  // the same for all warps
  if (__ldg(rp + n) - __ldg(rp) > kWide * n)
    na_rows<LOWER, 1>(n, rp, col, val, diag, rhs, x, err, lim_cycles);
  else
    na_rows<LOWER, kRows>(n, rp, col, val, diag, rhs, x, err, lim_cycles);
}

// Device address of the scratch array on the current device, looked up once
// per device (with that device current).
cudaError_t scratch_address(double **out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(g_mu);
  if (!g_scratch[dev]) {
    double *p = nullptr;
    e = cudaGetSymbolAddress((void **)&p, nle_noalloc_scratch);
    if (e != cudaSuccess) return e;
    g_scratch[dev] = p;
  }
  *out = g_scratch[dev];
  return cudaSuccess;
}

}  // namespace

namespace nle {
void set_global_error(const std::string &msg);
}

extern "C" nle_status nle_ic_apply_noalloc(int64_t n, const int32_t *Lrp, const int32_t *Lcol, const double *Lval,
                                           const int32_t *Urp, const int32_t *Ucol, const double *Uval,
                                           const double *diag, const double *g, double *c, void *stream) {
  if (n < 1 || n > kMaxN) {
    char buf[160];
    snprintf(buf, sizeof buf, "nle_ic_apply_noalloc: n = %lld is outside 1..%lld (the size of its fixed scratch)",
             (long long)n, (long long)kMaxN);
    nle::set_global_error(buf);
    return NLE_ERR_ARG;
  }
  if (!Lrp || !Lcol || !Lval || !Urp || !Ucol || !Uval || !diag || !g || !c) {
    nle::set_global_error("nle_ic_apply_noalloc: NULL pointer");
    return NLE_ERR_ARG;
  }
  {
    // c is written (with the not-yet-computed marker) before g is read, so
    // the two may not share memory
    const uintptr_t g0 = (uintptr_t)g, c0 = (uintptr_t)c, nb = (uintptr_t)n * sizeof(double);
    if (g0 < c0 + nb && c0 < g0 + nb) {
      nle::set_global_error("nle_ic_apply_noalloc: g and c overlap (in-place application is not supported)");
      return NLE_ERR_ARG;
    }
  }
  cudaStream_t s = (cudaStream_t)stream;
  double *z = nullptr;
  cudaError_t e = scratch_address(&z);
  if (e != cudaSuccess) {
    nle::set_global_error(std::string("nle_ic_apply_noalloc: cudaGetSymbolAddress: ") + cudaGetErrorString(e));
    return NLE_ERR_CUDA;
  }
  int *err = reinterpret_cast<int *>(z + kMaxN);
  int dev = 0, nsm = 0, coop = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  if (!coop) {
    nle::set_global_error("nle_ic_apply_noalloc: device lacks cooperative launch");
    return NLE_ERR_CUDA;
  }
  const long long lim = (long long)(2.0 * 2.1e9);  // ~2 s at the maximum SM clock
  // clear a launch error left pending by earlier work of the caller, so
  // that the check below reports this call's own launches
  (void)cudaGetLastError();
  k_na_fill<<<256, 256, 0, s>>>(z, c, n, err);
  e = cudaGetLastError();
  const int grid = (int)std::min<int64_t>(nsm, (n + kWarps - 1) / kWarps);  // one row a warp at least
  int64_t nn = n;
  const double *zc = z;
  void *fa[] = {&nn, (void *)&Lrp, (void *)&Lcol, (void *)&Lval, (void *)&diag, (void *)&g, (void *)&z, (void *)&err,
                (void *)&lim};
  void *ba[] = {&nn, (void *)&Urp, (void *)&Ucol, (void *)&Uval, (void *)&diag, (void *)&zc, (void *)&c, (void *)&err,
                (void *)&lim};
  if (e == cudaSuccess)
    e = cudaLaunchCooperativeKernel((void *)k_na_solve<true>, dim3(grid), dim3(32 * kWarps), fa, 0, s);
  if (e == cudaSuccess)
    e = cudaLaunchCooperativeKernel((void *)k_na_solve<false>, dim3(grid), dim3(32 * kWarps), ba, 0, s);
  int herr = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    nle::set_global_error(std::string("nle_ic_apply_noalloc: ") + cudaGetErrorString(e));
    return NLE_ERR_CUDA;
  }
  if (herr != 0) {
    nle::set_global_error(herr == NLE_ERR_CSR ? "nle_ic_apply_noalloc: an entry is not strictly triangular"
                                              : "nle_ic_apply_noalloc: a device wait ran out");
    return (nle_status)herr;
  }
  return NLE_OK;
}
