// Persistent cooperative kernels of the DACG-Newton eigensolver.
//
// One launch runs a whole phase on the device: DACG for eigenpair j
// (Section 4.1), the Newton iteration for eigenpair j with every inner PCG
// solve (Section 4.3, Algorithm 3.2), or one of the building blocks exposed
// for verification.  Passes over the vectors are separated by a bounded grid
// barrier; scalars are reduced deterministically so that every CTA takes the
// same control decisions without a host round trip.
//
// Algorithm 3.1 is applied in Gram form: with G_SR[s][t] = s_s^T r_t and
// G_QS[c][t] = q_c^T s_t (computed once per Newton step from the stored,
// rounded vectors), the two loops of Algorithm 3.1 reduce to k x k
// recurrences on scalars,
//   a_s = (s_s^T g - sum_{t>s} a_t G_SR[s][t]) / alpha_s,   w = g - R a,
//   c0  = Phat_0 w = L^{-T} L^{-1} w,
//   b_s = (r_s^T c0 - sum_{t<s} (a_t+b_t) G_SR[t][s]) / alpha_s,
//   z   = Q^T c0 - G_QS (a+b),   c = c0 - S (a+b) - Q z,
// which is algebraically identical to the paper's loop (same a_s, b_s, z)
// but needs one pass over S and R per dot-product group instead of 2k.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "nle_device.cuh"

namespace nle {

// ---------------------------------------------------------------------------
// small helpers over the chunks owned by a thread
// ---------------------------------------------------------------------------
// out[i][v] += sgn * sum_c coef[c] * X_c[row]   (X column c at X + c*ld),
// four columns per step for memory-level parallelism.
template <typename T, int RPC>
__device__ __forceinline__ void comb_add(const T *X, int64_t ld, int ncol, const double *coef, const int *slot,
                                         const Dev<T> &D, T (&out)[RPC][VT<T>::W], double sgn) {
  constexpr int W = VT<T>::W;
  const int64_t tid = gtid(), TT = gthreads();
  int c = 0;
  for (; c + 4 <= ncol; c += 4) {
    const T *col[4];
    T cf[4];
#pragma unroll
    for (int u = 0; u < 4; u++) {
      col[u] = X + (int64_t)(slot ? slot[c + u] : c + u) * ld;
      cf[u] = T(sgn * coef[c + u]);
    }
#pragma unroll
    for (int i = 0; i < RPC; i++) {
      const int64_t ch = tid + i * TT;
      if (ch < D.nchunks) {
        T q[4][W];
#pragma unroll
        for (int u = 0; u < 4; u++) ldc(col[u] + ch * W, q[u]);
#pragma unroll
        for (int u = 0; u < 4; u++)
#pragma unroll
          for (int v = 0; v < W; v++) out[i][v] += cf[u] * q[u][v];
      }
    }
  }
  for (; c < ncol; c++) {
    const T cf = T(sgn * coef[c]);
    const T *cl = X + (int64_t)(slot ? slot[c] : c) * ld;
#pragma unroll
    for (int i = 0; i < RPC; i++) {
      const int64_t ch = tid + i * TT;
      if (ch < D.nchunks) {
        T q[W];
        ldc(cl + ch * W, q);
#pragma unroll
        for (int v = 0; v < W; v++) out[i][v] += cf * q[v];
      }
    }
  }
}

// slot0 + c: sum over owned rows of X_c[row] * val[i][v], for each column c.
// Four columns per step so that 4*RPC independent loads are in flight.
template <typename T, int RPC>
__device__ __forceinline__ void dots_put(Shared &sh, int slot0, const T *X, int64_t ld, int ncol, const int *slot,
                                         const Dev<T> &D, const T (&val)[RPC][VT<T>::W], bool reverse) {
  constexpr int W = VT<T>::W;
  const int64_t tid = gtid(), TT = gthreads();
  int c = 0;
  for (; c + 4 <= ncol; c += 4) {
    const T *col[4];
#pragma unroll
    for (int u = 0; u < 4; u++) col[u] = X + (int64_t)(slot ? slot[c + u] : c + u) * ld;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int i = 0; i < RPC; i++) {
      const int64_t k = tid + i * TT;
      const int64_t ch = reverse ? D.nchunks - 1 - k : k;
      if (k < D.nchunks) {
        T q[4][W];
#pragma unroll
        for (int u = 0; u < 4; u++) ldc(col[u] + ch * W, q[u]);
#pragma unroll
        for (int u = 0; u < 4; u++)
#pragma unroll
          for (int v = 0; v < W; v++) acc[u] += wide(q[u][v]) * wide(val[i][v]);
      }
    }
#pragma unroll
    for (int u = 0; u < 4; u++) red_put(sh, slot0 + c + u, acc[u]);
  }
  for (; c < ncol; c++) {
    const T *cl = X + (int64_t)(slot ? slot[c] : c) * ld;
    double acc = 0.0;
#pragma unroll
    for (int i = 0; i < RPC; i++) {
      const int64_t k = tid + i * TT;
      const int64_t ch = reverse ? D.nchunks - 1 - k : k;
      if (k < D.nchunks) {
        T q[W];
        ldc(cl + ch * W, q);
#pragma unroll
        for (int v = 0; v < W; v++) acc += wide(q[v]) * wide(val[i][v]);
      }
    }
    red_put(sh, slot0 + c, acc);
  }
}

template <typename T, int RPC>
__device__ __forceinline__ double self_dot(const T (&a)[RPC][VT<T>::W], const T (&b)[RPC][VT<T>::W]) {
  double acc = 0.0;
#pragma unroll
  for (int i = 0; i < RPC; i++)
#pragma unroll
    for (int v = 0; v < VT<T>::W; v++) acc += wide(a[i][v]) * wide(b[i][v]);
  return acc;
}

// ---------------------------------------------------------------------------
// Gram form of Algorithm 3.1: scalar recurrences (one thread, every CTA)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void coef_a(Shared &sh, int k) {
  if (threadIdx.x == 0) {
    for (int s = k - 1; s >= 0; s--) {
      double t = sh.sg[s];
      for (int u = s + 1; u < k; u++) t -= sh.a[u] * sh.gsr[s][u];
      sh.a[s] = t / sh.alpha[s];
    }
  }
  __syncthreads();
}

// rc[t] = r_t^T c0 (chronological), qc[c] = q_c^T c0
__device__ __forceinline__ void coef_b(Shared &sh, int k, int m, const double *rc, const double *qc) {
  if (threadIdx.x == 0) {
    for (int s = 0; s < k; s++) {
      double t = rc[s];
      for (int u = 0; u < s; u++) t -= sh.ab[u] * sh.gsr[u][s];
      sh.b[s] = t / sh.alpha[s];
      sh.ab[s] = sh.a[s] + sh.b[s];
    }
    for (int c = 0; c < m; c++) {
      double t = qc[c];
      for (int u = 0; u < k; u++) t -= sh.ab[u] * sh.gqs[c][u];
      sh.zq[c] = t;
    }
  }
  __syncthreads();
}

// Gram matrices of the stored pairs: gsr[s][t] = s_s^T r_t, gqs[c][t] = q_c^T s_t.
template <typename T, int RPC>
__device__ bool gram(const Dev<T> &D, Shared &sh, Ctl &ctl, int m, int k) {
  constexpr int W = VT<T>::W;
  if (k == 0) return true;
  const int64_t tid = gtid(), TT = gthreads();
  const int per_s = k + m;  // slots per pair
  const int smax = RED_MAX / per_s;
  for (int s0 = 0; s0 < k; s0 += smax) {
    const int s1 = min(k, s0 + smax);
    for (int s = s0; s < s1; s++) {
      T sv[RPC][W];
      const T *scol = D.S + (int64_t)sh.order[s] * D.npad;
#pragma unroll
      for (int i = 0; i < RPC; i++) {
        const int64_t ch = tid + i * TT;
        if (ch < D.nchunks)
          ldc(scol + ch * W, sv[i]);
        else
#pragma unroll
          for (int v = 0; v < W; v++) sv[i][v] = T(0);
      }
      dots_put<T, RPC>(sh, (s - s0) * per_s, D.R, D.npad, k, sh.order, D, sv, false);
      dots_put<T, RPC>(sh, (s - s0) * per_s + k, D.Q, D.npad, m, nullptr, D, sv, false);
    }
    if (!reduce_all(D, sh, ctl, (s1 - s0) * per_s, 10)) return false;
    if (threadIdx.x == 0)
      for (int s = s0; s < s1; s++) {
        for (int t = 0; t < k; t++) sh.gsr[s][t] = sh.sc[(s - s0) * per_s + t];
        for (int c = 0; c < m; c++) sh.gqs[c][s] = sh.sc[(s - s0) * per_s + k + c];
      }
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int s = 0; s < k; s++) sh.alpha[s] = sh.gsr[s][s];
  __syncthreads();
  return true;
}

// ---------------------------------------------------------------------------
// preconditioner tail: forward solve on w = g - R a, backward solve, the dot
// products of Algorithm 3.1's forward loop and Gram-Schmidt, and the output
// pass out = c0 - S(a+b) - Q z (+ beta * out, beta = gamma'/gamma_old when
// use_beta).  On entry z/c0 hold the not-yet-computed marker and the solve
// queues are reset.  *gamma_new receives gamma' = g^T c.
//
// The triangular solves (trsv_block) work slab by slab, one slab per CTA,
// with ctl.twarps warps of the CTA taking the slab's rows in order.  Dynamic
// shared memory holds two slab-sized buffers: A receives the forward results
// z of the slab, B first holds the forward right-hand side w and then the
// backward results; no right-hand side is fetched from global memory on the
// dependency chain.
// ---------------------------------------------------------------------------
extern __shared__ __align__(16) unsigned char nle_dyn_smem[];  // two slabs of the triangular solves

// Triangular solves compiled into this translation unit: 0 the level schedule
// with both forms, 1 the chain schedule, 2 the level schedule's polled form alone
// (the build compiles every (precision, rows-per-thread) pair once for each, so
// that the chain and the polled solves keep their registers); the kernels carry
// it as a template argument so that the builds' kernels have distinct names.
#ifndef NLE_TRSV_TU
#define NLE_TRSV_TU 0
#endif
constexpr bool kChainTU = NLE_TRSV_TU == 1, kStepTU = NLE_TRSV_TU == 0;

// ---------------------------------------------------------------------------
// Step form of the level schedule, one solve slab of rows per CTA.
//
// Solving a slab is a chain of levels, a few rows to a few dozen each, so what
// counts is the time from one level to the next, and nothing on that path may
// wait on global memory.
//  * The first warps solve, taking the slab's steps (plan_steps) in turn: up to
//    32 rows of one level.  All operands come from the slab's shared-memory
//    window, results go to the window and, for the other slabs, to global
//    memory.  A warp has the coefficients and operand addresses of its step
//    in registers (loaded while the others work) when the level before ends:
//    the warps of that level's steps arrive at a named barrier on which the
//    warp of the next level's first step waits, and that one releases the
//    next step of its level, and so on.  (A level with more steps than warps
//    joins through reports in sh.fin instead.)
//  * COPY_WARPS warps copy the halo, the values the slab needs from other
//    slabs, from global memory into the window as they are published (a
//    value is its own ready flag), and publish the first value of their share
//    still missing.  A step states how many halo values it and the steps
//    before it need, and its warp waits for them before it takes over.
// A value takes about 1 us from one slab to the next, as long as some eight
// levels, so a solve slab is several slabs (and fewer CTAs solve) where the
// levels are narrow.
//
// Every wait ends: the steps of a slab follow the level order, and the halo
// values listed up to a step belong to rows of lower levels than that step's,
// so the unfinished row of lowest level always gets its inputs; all CTAs are
// resident (cooperative launch).  The waits on flags are also bounded in
// time; past the bound the warps go on without waiting, so that every warp
// takes all its steps and the barriers between the warps always complete.
// Barriers and votes need whole warps: what decides a wait is the same value
// in all lanes, and the warp converges before them.
//
// Sums are formed as the 8-lane (16-lane) reduction of trsv_block forms them:
// entry k of a row in partial sum k mod 8 (16), each partial sum in ascending
// k, the partial sums added pairwise in the order of its butterfly, so both
// forms give the same bits (the sign of a zero aside).  With LPR lanes per row, lane g holds the partial
// sums p with p mod LPR = g: the first additions are in the lane, the others
// between lanes.  FP32: one (two) lanes, since a shuffle costs as much as six
// additions.  FP64: four, since an FP64 instruction occupies its quarter of
// the SM for 64 cycles whatever the number of lanes (measured: 64 cycles for
// one warp, 256 for four instructions, dependent or not).
// ---------------------------------------------------------------------------
// Waits until the slab's steps from `from` up to `last` have reported their
// end.  Step x of a warp is done when its next one (x + number of warps) has
// begun, so the 32 steps up to `last` are enough.  Bounded.
__device__ __forceinline__ void await_steps(const Shared &sh, int from, int last, long long spin_ns, State *st) {
  const int x = last - (int)(threadIdx.x & 31);
  const volatile int *f = &sh.fin[x & 63];
  long long t0 = 0;
  for (int it = 1;; it++) {
    if (__all_sync(0xffffffffu, x < from || *f > x)) break;
    if ((it & 4095) == 0 && __any_sync(0xffffffffu, wait_over(st, t0, spin_ns, 105))) break;
  }
  __threadfence_block();
}

// Waits until `need` halo values have arrived; returns how many have (the
// same value in all lanes).  Bounded.
__device__ __forceinline__ int await_halo(const Shared &sh, int need, long long spin_ns, State *st) {
  const unsigned arrived = smem_addr(&sh.arrived[0]);
  long long t0 = 0;
  for (int it = 1;; it++) {
    const int4 f = lds4(arrived);
    const int here = (int)__reduce_min_sync(0xffffffffu, (unsigned)min(min(f.x, f.y), min(f.z, f.w)));
    if (need <= here) {
      __threadfence_block();
      return here;
    }
    if ((it & 4095) == 0 && __any_sync(0xffffffffu, wait_over(st, t0, spin_ns, 102))) return 0x7fffffff;
  }
}

// Barrier w + 1 belongs to warp w (0 is __syncthreads).  The warp converges
// first: a barrier counts whole warps each time it is executed.
__device__ __forceinline__ void bar_wait(int id, int threads) {
  __syncwarp();
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
  __syncwarp();
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// End of a step: the barriers its head names (n of them from that of warp w).
struct StepEnd {
  int n, bar, threads;
  __device__ __forceinline__ explicit StepEnd(int sync)
      : n(sync >> 14 & 15), bar((sync >> 10 & 15) + 1), threads(sync >> 18 & 1023) {}
  __device__ __forceinline__ void arrive(int nwarp) const {
    __syncwarp();
    if (n > 0) asm volatile("bar.arrive %0, %1;" ::"r"(bar), "r"(threads) : "memory");
    if (__builtin_expect(n > 1, 0))
      for (int i = 1, w = bar; i < n; i++) {
        w = w == nwarp ? 1 : w + 1;
        asm volatile("bar.arrive %0, %1;" ::"r"(w), "r"(threads) : "memory");
      }
  }
};

__device__ __forceinline__ void report_end(Shared &sh, int step) {
  if ((threadIdx.x & 31) == 0) {
    __threadfence_block();
    sts(smem_addr(&sh.fin[step & 63]), step + 1);
  }
}

// One triangular solve of the calling CTA: rows [b0, b0 + rows) of z or c0.
// The window, from the start of dynamic shared memory: `rows` own results,
// the zero, the halo.  The solves are inlined and read the problem's pointers
// where they are used (from the constant bank, the descriptor being a kernel
// parameter): copies of them, or a call, cost registers or reloads inside
// the loop (inlined against called: a chain of single rows 0.53 / 0.81 ms, two
// eigenpairs of 100^3 mixed 482 / 647 ms, a batch of 48 graphs 498 / 556 ms, an FP64 application
// of 60 x 70 309 / 305 us).
template <bool LOWER, typename T>
__device__ __forceinline__ const TriSteps<T> &steps_of(const Dev<T> &D) {
  if constexpr (LOWER) return D.SL;
  else return D.SU;
}

template <typename T>
__device__ __forceinline__ void steps_begin(const Dev<T> &D, Shared &sh) {
  if (threadIdx.x < COPY_WARPS) sh.arrived[threadIdx.x] = 32 * threadIdx.x;  // first value of its share
  if (threadIdx.x < 64) sh.fin[threadIdx.x] = 0;
  if (threadIdx.x == 0) reinterpret_cast<T *>(nle_dyn_smem)[D.bsize * D.steps] = T(0);
  __syncthreads();
}

// The copying warps of a step solve.
template <bool LOWER, typename T>
__device__ __forceinline__ void steps_copy(const Dev<T> &D, Shared &sh, long long spin_ns) {
  const int m = (int)(threadIdx.x >> 5) - (NWARP - COPY_WARPS);
  if (m < 0) return;
  const TriSteps<T> &M = steps_of<LOWER>(D);
  const int h0 = __ldg(M.hptr + grank()), h1 = __ldg(M.hptr + grank() + 1);
  copy_halo<T>(M.hpos + h0, h1 - h0, m, LOWER ? D.z : D.c0,
               smem_addr(nle_dyn_smem) + (unsigned)((D.bsize * D.steps + 1) * (int)sizeof(T)), sh, spin_ns, D.st);
}

// keeps the computation of a register where it is written: the compiler moves
// loads, selects and address sums down to their first use otherwise, behind
// the barrier that begins a step
__device__ __forceinline__ void pin(unsigned &v) { asm volatile("" : "+r"(v)); }
__device__ __forceinline__ void pin(float &v) { asm volatile("" : "+f"(v)); }
__device__ __forceinline__ void pin(double &v) { asm volatile("" : "+d"(v)); }

// two FP32 operations per instruction, each rounded as the single one
using F2 = float2;
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 d;
  asm("{.reg .b64 x, y, z, w;\nmov.b64 x, {%2, %3};\nmov.b64 y, {%4, %5};\nmov.b64 z, {%6, %7};\n"
      "fma.rn.f32x2 w, x, y, z;\nmov.b64 {%0, %1}, w;}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
  F2 d;
  asm("{.reg .b64 x, y, w;\nmov.b64 x, {%2, %3};\nmov.b64 y, {%4, %5};\nmul.rn.f32x2 w, x, y;\nmov.b64 {%0, %1}, w;}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
  F2 d;
  asm("{.reg .b64 x, y, w;\nmov.b64 x, {%2, %3};\nmov.b64 y, {%4, %5};\nadd.rn.f32x2 w, x, y;\nmov.b64 {%0, %1}, w;}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}

// Partial sums of a lane: NP of them, entry e of the lane in sum e mod NP.
template <typename T, int NP>
struct Sums;
template <>
struct Sums<float, 8> {
  F2 acc[4];
  template <int E>
  __device__ __forceinline__ void start(const float (&a)[E], const float (&v)[E]) {
#pragma unroll
    for (int j = 0; j < 4; j++) acc[j] = mul2(F2{a[2 * j], a[2 * j + 1]}, F2{v[2 * j], v[2 * j + 1]});
#pragma unroll
    for (int e = 8; e < E; e += 2) acc[e / 2 & 3] = fma2(F2{a[e], a[e + 1]}, F2{v[e], v[e + 1]}, acc[e / 2 & 3]);
  }
  // the lane's quad i
  __device__ __forceinline__ void quad(int i, const float (&a)[4], const float (&v)[4]) {
#pragma unroll
    for (int e = 0; e < 4; e += 2) {
      const F2 x{a[e], a[e + 1]}, y{v[e], v[e + 1]};
      if (i & 1) acc[2 + e / 2] = fma2(x, y, acc[2 + e / 2]);
      else acc[e / 2] = fma2(x, y, acc[e / 2]);
    }
  }
  __device__ __forceinline__ float total() const {
    const F2 s = add2(add2(acc[0], acc[2]), add2(acc[1], acc[3]));
    return s.x + s.y;
  }
};
// Every FP64 product goes into an fma and every other sum is an explicit add: of two
// products that meet in one sum the compiler picks the one it rounds, and rows of more
// than 8 entries differed from trsv_block's in the last bit.
template <>
struct Sums<double, 2> {
  double acc[2];
  template <int E>
  __device__ __forceinline__ void start(const double (&a)[E], const double (&v)[E]) {
    acc[0] = acc[1] = 0.0;
#pragma unroll
    for (int e = 0; e < E; e++) acc[e & 1] = fma(a[e], v[e], acc[e & 1]);
  }
  __device__ __forceinline__ void quad(int, const double (&a)[4], const double (&v)[4]) {
#pragma unroll
    for (int e = 0; e < 4; e++) acc[e & 1] = fma(a[e], v[e], acc[e & 1]);
  }
  __device__ __forceinline__ double total() const { return __dadd_rn(acc[0], acc[1]); }
};

// LPR lanes per row, E entries of a lane held in registers (2 or quads; all of
// them are summed, padding too: a predicated FP64 instruction costs as much).
template <bool LOWER, int LPR, int E, typename T>
__device__ __forceinline__ void trsv_steps(const Dev<T> &D, const T *rhs_all, Shared &sh, long long spin_ns) {
  constexpr int PER = 32 / LPR, NP = sizeof(T) == 8 ? 2 : 8, C = E < 4 ? E : 4;
  constexpr unsigned TS = sizeof(T);
  const int64_t b0 = (int64_t)grank() * D.bsize * D.steps;
  if (b0 >= D.npad) return;  // a CTA past the last solve slab
  const TriSteps<T> &M = steps_of<LOWER>(D);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned w0 = smem_addr(nle_dyn_smem), zero = w0 + TS * (unsigned)(D.bsize * D.steps);
  steps_begin(D, sh);
  if (warp < D.step_warps) {
    const int s0 = __ldg(M.step0 + grank()), ns = __ldg(M.step0 + grank() + 1) - s0;
    const int4 *heads = reinterpret_cast<const int4 *>(M.head + s0);
    const int32_t *rows = M.row + (int64_t)s0 * PER + lane / LPR;
    const int nwarp = D.step_warps, next = warp + 1 == nwarp ? 1 : warp + 2;
    const T *rhs = rhs_all + b0, *rdiag = D.rdiag + b0;
    T *x = (LOWER ? D.z : D.c0) + b0;
    unsigned c[E], own = 0;
    T a[E], b = T(0), rdg = T(1);
    int rl = 0;
    auto head = [&](int t) { return t < ns ? __ldg(heads + 2 * t) : make_int4(0, 0, 0, 0); };
    auto row_of = [&](int t) { return t < ns ? __ldg(rows + t * PER) : 0; };
    // lanes past the step's repeat its last row (and store the same result)
    auto lane_of = [&](int lanes) {
      return LPR == 1 ? min(lane, lanes - 1) : lane < lanes ? lane : lanes - LPR + (lane & (LPR - 1));
    };
    // the step's coefficients, operands, right-hand side and pivot
    auto fetch = [&](const int4 &H, int row) {
      rl = row;
      const int lanes = H.z & 63, n = H.z >> 6 & 1023;
      const int32_t *po = M.opnd + 4 * ((int64_t)H.x + lane_of(lanes));
      const T *pv = M.val + 4 * ((int64_t)H.x + lane_of(lanes));
#pragma unroll
      for (int i = 0; i < E; i += C) {
        int ci[C] = {};
        T ai[C] = {};
        if (i < n) {
          ldr(po + i * lanes, ci);
          ldr(pv + i * lanes, ai);
        }
#pragma unroll
        for (int e = 0; e < C; e++) c[i + e] = i < n ? w0 + (unsigned)ci[e] : zero, a[i + e] = ai[e];
      }
      rdg = __ldg(rdiag + rl);
      b = __ldcg(rhs + rl);
      own = w0 + TS * rl;
      // all of it is in registers before the warp waits for its turn
#pragma unroll
      for (int e = 0; e < E; e++) pin(c[e]), pin(a[e]);
      pin(rdg), pin(b), pin(own);
    };
    int t = warp;
    // heads and rows two turns ahead, so that a fetch waits for one load only
    int4 H = head(t), N = head(t + nwarp);
    int nrow = row_of(t + nwarp);
    if (t < ns) fetch(H, row_of(t));
    int here = 0;  // halo values known to have arrived
    for (; t < ns; t += nwarp) {
      const unsigned flags = (unsigned)H.z >> 16;
      const int n = H.z >> 6 & 1023, threads = H.y & 1023;
      const bool plain = flags == 0 && n <= E;  // nothing special, all entries in registers
      const StepEnd end(H.y);
      __syncwarp();
      if (H.w > here) here = await_halo(sh, H.w, spin_ns, D.st);
      if (threads) bar_wait(warp + 1, threads);
      if (__builtin_expect(!plain, 0)) {
        if ((flags & STEP_EARLY) && nwarp > 1) bar_arrive(next, 64);
        if (flags & STEP_WAIT) {
          const int4 H2 = __ldg(heads + 2 * t + 1);
          await_steps(sh, H2.y, H2.x - 1, spin_ns, D.st);
        }
      }
      T v[E];
#pragma unroll
      for (int e = 0; e < E; e++) lds(c[e], v[e]);
      Sums<T, NP> S;
      S.start(a, v);
      if (__builtin_expect(!plain, 0)) {
        const int lanes = H.z & 63;
#pragma unroll 1
        for (int i = (E + 3) / 4; 4 * i < n; i++) {  // quads past the ones in registers
          const int64_t at = 4 * ((int64_t)H.x + lane_of(lanes) + (int64_t)i * lanes);
          int ci[4];
          T ai[4], vi[4];
          ldr(M.opnd + at, ci);
          ldr(M.val + at, ai);
#pragma unroll
          for (int e = 0; e < 4; e++) lds(w0 + (unsigned)ci[e], vi[e]);
          S.quad(i, ai, vi);
        }
      }
      T sum = S.total();
#pragma unroll
      for (int o = LPR / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      const T val = (b - sum) * rdg;
      sts(own, val);
      end.arrive(nwarp);
      st_relaxed(x + rl, val);
      if (flags & STEP_REPORT) {
        __syncwarp();
        report_end(sh, t);
      }
      H = N;
      if (t + nwarp < ns) fetch(H, nrow);
      N = head(t + 2 * nwarp);
      nrow = row_of(t + 2 * nwarp);
    }
  }
  steps_copy<LOWER>(D, sh, spin_ns);
  __syncthreads();
}

// The step form of the forward (LOWER) or backward solve with right-hand side
// rhs (global memory).
template <bool LOWER, typename T>
__device__ __forceinline__ void steps_solve(const Dev<T> &D, Shared &sh, const Ctl &ctl, const T *rhs) {
  if constexpr (sizeof(T) == 8) {
    if (D.step_n <= 2) trsv_steps<LOWER, 4, 2, T>(D, rhs, sh, ctl.spin_ns);
    else trsv_steps<LOWER, 4, 4, T>(D, rhs, sh, ctl.spin_ns);
  } else if (D.trows == 2) {
    if (D.step_n <= 16) trsv_steps<LOWER, 2, 16, T>(D, rhs, sh, ctl.spin_ns);
    else trsv_steps<LOWER, 2, 24, T>(D, rhs, sh, ctl.spin_ns);
  } else {
    if (D.step_n <= 8) trsv_steps<LOWER, 1, 8, T>(D, rhs, sh, ctl.spin_ns);
    else trsv_steps<LOWER, 1, 16, T>(D, rhs, sh, ctl.spin_ns);
  }
}

template <typename T>
__device__ __forceinline__ bool trsv_forward(const Dev<T> &D, Shared &sh, Ctl &ctl, int k) {
  if constexpr (kStepTU) {
    if (D.steps) {
      if (k == 0) {
        steps_solve<true, T>(D, sh, ctl, D.g);
        return true;
      }
      // w = g - R a (in y, which holds nothing needed any more)
      constexpr int W = VT<T>::W;
      const int64_t TT = gthreads();
      for (int64_t ch = gtid(); ch < D.nchunks; ch += TT) {
        T w[W];
        ldc(D.g + ch * W, w);
        for (int t = 0; t < k; t++) {
          T r[W];
          ldc(D.R + (int64_t)sh.order[t] * D.npad + ch * W, r);
#pragma unroll
          for (int v = 0; v < W; v++) w[v] -= T(sh.a[t]) * r[v];
        }
        stv(D.y + ch * W, w);
      }
      if (!grid_sync(D.st, sh, ctl, 20)) return false;
      steps_solve<true, T>(D, sh, ctl, D.y);
      return true;
    }
  }
  const TriEll<T> L{D.Loff, D.Lw, D.Lcol, D.Lval, D.rdiag, D.Lround, D.trows};
  T *bufA = reinterpret_cast<T *>(nle_dyn_smem);
  T *bufB = bufA + D.bsize;
  const int64_t b0 = (int64_t)grank() * D.bsize;
  const int64_t nb = max((int64_t)0, min(D.npad, b0 + D.bsize) - b0);
  // w = g - R a for the slab's rows (trsv_block's first barrier orders these
  // stores before any use)
  for (int64_t i = threadIdx.x; i < nb; i += blockDim.x) {
    T w = __ldcg(D.g + b0 + i);
    for (int t = 0; t < k; t++) w -= T(sh.a[t]) * __ldcg(D.R + (int64_t)sh.order[t] * D.npad + b0 + i);
    bufB[i] = w;
  }
  if constexpr (kChainTU) {
    const TriChain<T> C{D.Loff, D.Lw, D.Lcol, D.Lval, D.rdiag, D.Lwp, D.Ltask};
    trsv_chain<true, T>(C, D.z, D.npad, D.bsize, ctl.spin_ns, ctl.poll_ns, D.st, bufA,
                        [&](int64_t r) { return bufB[r - b0]; });
  } else {
    trsv_block<true, T>(L, D.z, D.npad, D.bsize, ctl.twarps, ctl.spin_ns, ctl.poll_ns, D.st, bufA,
                        [&](int64_t r) { return bufB[r - b0]; });
  }
  return true;
}

// The right-hand side of the backward solve is the forward result of the
// CTA's own slab (buffer A, or z in the step form), complete after
// trsv_forward's closing __syncthreads, so no grid barrier separates the two
// solves.
template <typename T>
__device__ __forceinline__ void trsv_backward(const Dev<T> &D, Shared &sh, const Ctl &ctl) {
  if constexpr (kStepTU) {
    if (D.steps) {
      steps_solve<false, T>(D, sh, ctl, D.z);
      return;
    }
  }
  const TriEll<T> U{D.Uoff, D.Uw, D.Ucol, D.Uval, D.rdiag, D.Uround, D.trows};
  const T *bufA = reinterpret_cast<const T *>(nle_dyn_smem);
  T *bufB = reinterpret_cast<T *>(nle_dyn_smem) + D.bsize;
  const int64_t b0 = (int64_t)grank() * D.bsize;
  if constexpr (kChainTU) {
    const TriChain<T> C{D.Uoff, D.Uw, D.Ucol, D.Uval, D.rdiag, D.Uwp, D.Utask};
    trsv_chain<false, T>(C, D.c0, D.npad, D.bsize, ctl.spin_ns, ctl.poll_ns, D.st, bufB,
                         [&](int64_t r) { return bufA[r - b0]; });
  } else {
    trsv_block<false, T>(U, D.c0, D.npad, D.bsize, ctl.twarps, ctl.spin_ns, ctl.poll_ns, D.st, bufB,
                         [&](int64_t r) { return bufA[r - b0]; });
  }
}

template <typename T>
__device__ __forceinline__ void reset_queues(const Dev<T> &D) {
  if (lead_cta() && threadIdx.x == 0) {
    D.st->qf = 0u;
    D.st->qb = 0u;
  }
}

template <typename T, int RPC>
__device__ bool precond_tail(const Dev<T> &D, Shared &sh, Ctl &ctl, int m, int k, T *out, double gamma_old,
                             bool use_beta, double *gamma_new) {
  constexpr int W = VT<T>::W;
  const int64_t tid = gtid(), TT = gthreads();
  if (!trsv_forward<T>(D, sh, ctl, k)) return false;
  tmark(sh, PH_FWD);
  trsv_backward<T>(D, sh, ctl);
  if (!grid_sync(D.st, sh, ctl, 21)) return false;
  tmark(sh, PH_BWD);
  // dot products of c0: slots [0,k) r_t^T c0 ; k: g^T c0 ; [k+1, k+1+m) q_c^T c0
  T cv[RPC][W];
  {
    double acc = 0.0;
#pragma unroll
    for (int i = 0; i < RPC; i++) {
      const int64_t ch = tid + i * TT;
      if (ch < D.nchunks) {
        T gg[W];
        ldc(D.c0 + ch * W, cv[i]);
        ldc(D.g + ch * W, gg);
#pragma unroll
        for (int v = 0; v < W; v++) acc += double(gg[v]) * double(cv[i][v]);
      } else {
#pragma unroll
        for (int v = 0; v < W; v++) cv[i][v] = T(0);
      }
    }
    red_put(sh, k, acc);
    dots_put<T, RPC>(sh, 0, D.R, D.npad, k, sh.order, D, cv, false);
    dots_put<T, RPC>(sh, k + 1, D.Q, D.npad, m, nullptr, D, cv, false);
  }
  if (!reduce_all(D, sh, ctl, k + 1 + m, 22)) return false;
  tmark(sh, PH_DOTS);
  const double gc0 = sh.sc[k];
  coef_b(sh, k, m, sh.sc, sh.sc + k + 1);
  // gamma' = g^T c = g^T c0 - (S^T g)(a+b)   (g is orthogonal to Q)
  double gnew = gc0;
  for (int s = 0; s < k; s++) gnew -= sh.sg[s] * sh.ab[s];
  *gamma_new = gnew;
  const double beta = use_beta ? gnew / gamma_old : 0.0;
  // output pass: out = c0 - S ab - Q z + beta*out
  {
    if (k > 0) comb_add<T, RPC>(D.S, D.npad, k, sh.ab, sh.order, D, cv, -1.0);
    if (m > 0) comb_add<T, RPC>(D.Q, D.npad, m, sh.zq, nullptr, D, cv, -1.0);
#pragma unroll
    for (int i = 0; i < RPC; i++) {
      const int64_t ch = tid + i * TT;
      if (ch < D.nchunks) {
        if (use_beta) {
          T po[W];
          ldc(out + ch * W, po);
#pragma unroll
          for (int v = 0; v < W; v++) cv[i][v] += T(beta) * po[v];
        }
        stv(out + ch * W, cv[i]);
      }
    }
  }
  const bool ok = grid_sync(D.st, sh, ctl, 23);
  tmark(sh, PH_DIR);
  return ok;
}

// ---------------------------------------------------------------------------
// PCG on the correction equation (Section 4.3): J s = -r, s perp Q, with
// J = (I-QQ^T)(A - theta I)(I-QQ^T) and P_k by Algorithm 3.1.
// Inputs in device memory: rT (r in working precision), Q (m columns), the
// k stored pairs (sh.order, S, R) and their Gram matrices (sh.gsr, sh.gqs,
// sh.alpha).  Output: s.  The residual g is kept orthogonal to Q by
// g <- g - alpha (y - Q (Q^T y)), which equals the update followed by the
// projection of g when g is orthogonal to Q.
// ---------------------------------------------------------------------------
struct PcgOut {
  int its;
  int exit;
  double rs;  // r^T s at exit (= alpha of the new pair)
  double g0, gn, eres;
};

template <typename T, int RPC>
__device__ bool pcg_solve(const Dev<T> &D, const Opts &O, Shared &sh, Ctl &ctl, int m, int k, double theta,
                          int max_pcg, PcgOut &res) {
  constexpr int W = VT<T>::W;
  const int64_t tid = gtid(), TT = gthreads();
  const T Tsent = sentinel<T>();
  T gv[RPC][W];
  // --- initial residual g = -(I - QQ^T) r, s = 0
  {
    T rv[RPC][W];
#pragma unroll
    for (int i = 0; i < RPC; i++) {
      const int64_t ch = tid + i * TT;
      if (ch < D.nchunks)
        ldc(D.rT + ch * W, rv[i]);
      else
#pragma unroll
        for (int v = 0; v < W; v++) rv[i][v] = T(0);
    }
    dots_put<T, RPC>(sh, 0, D.Q, D.npad, m, nullptr, D, rv, false);
    if (!reduce_all(D, sh, ctl, m, 30)) return false;
    for (int c = threadIdx.x; c < m; c += TPB) sh.qv[c] = -sh.sc[c];
    __syncthreads();
    comb_add<T, RPC>(D.Q, D.npad, m, sh.qv, nullptr, D, rv, 1.0);  // rv = r - Q Q^T r
    T sent[W], zero[W];
#pragma unroll
    for (int v = 0; v < W; v++) sent[v] = Tsent, zero[v] = T(0);
#pragma unroll
    for (int i = 0; i < RPC; i++) {
      const int64_t ch = tid + i * TT;
#pragma unroll
      for (int v = 0; v < W; v++) gv[i][v] = -rv[i][v];
      if (ch < D.nchunks) {
        stv(D.g + ch * W, gv[i]);
        stv(D.s + ch * W, zero);
        stv(D.z + ch * W, sent);
        stv(D.c0 + ch * W, sent);
      }
    }
    reset_queues(D);
    red_put(sh, 0, self_dot<T, RPC>(gv, gv));
    dots_put<T, RPC>(sh, 1, D.S, D.npad, k, sh.order, D, gv, false);
    if (!reduce_all(D, sh, ctl, 1 + k, 31)) return false;
    tmark(sh, PH_UPDATE);
  }
  const double g0 = sqrt(sh.sc[0]);
  if (threadIdx.x == 0)
    for (int s = 0; s < k; s++) sh.sg[s] = sh.sc[1 + s];
  __syncthreads();
  double gamma = 0.0;
  res.g0 = g0;
  res.gn = g0;
  res.eres = 0.0;
  res.rs = 0.0;
  res.exit = 1;  // NLE_EXIT_MAXIT
  res.its = 0;
  double gprev = g0, eprev = 0.0;
  for (int l = 0; l < max_pcg; l++) {
    // direction p = P_k g + beta p (one copy of the solves' code for the first
    // direction and the others)
    coef_a(sh, k);
    {
      double gnew;
      if (!precond_tail<T, RPC>(D, sh, ctl, m, k, D.p, gamma, l > 0, &gnew)) return false;
      gamma = gnew;
    }
    // --- pass A: y = (A - theta I) p, delta = p^T y, Q^T y
    T yv[RPC][W];
    {
      double pty = 0.0;
#pragma unroll
      for (int i = 0; i < RPC; i++) {
        const int64_t ch = tid + i * TT;
        if (ch < D.nchunks) {
          T acc[W], pp[W];
          sell_rows<W, T, T, T>(D.A, D.p, ch, acc);
          ldc(D.p + ch * W, pp);
#pragma unroll
          for (int v = 0; v < W; v++) {
            yv[i][v] = acc[v] - T(theta) * pp[v];
            pty += double(pp[v]) * double(yv[i][v]);
          }
          stv(D.y + ch * W, yv[i]);
        } else {
#pragma unroll
          for (int v = 0; v < W; v++) yv[i][v] = T(0);
        }
      }
      red_put(sh, 0, pty);
      dots_put<T, RPC>(sh, 1, D.Q, D.npad, m, nullptr, D, yv, false);
      if (!reduce_all(D, sh, ctl, 1 + m, 32)) return false;
      tmark(sh, PH_SPMV);
    }
    const double delta = sh.sc[0];
    if (!(delta > 0.0)) {
      res.exit = 4;  // NLE_EXIT_BREAKDOWN
      res.its = l;
      break;
    }
    res.its = l + 1;
    const double alpha = gamma / delta;
    // --- pass B: s += alpha p; g -= alpha (y - Q Q^T y); exit scalars; S^T g
    {
      for (int c = threadIdx.x; c < m; c += TPB) sh.qv[c] = -sh.sc[1 + c];
      __syncthreads();
      comb_add<T, RPC>(D.Q, D.npad, m, sh.qv, nullptr, D, yv, 1.0);  // yv = (I - QQ^T) y
      double rs = 0.0, sg = 0.0, ss = 0.0;
      T sent[W];
#pragma unroll
      for (int v = 0; v < W; v++) sent[v] = Tsent;
#pragma unroll
      for (int i = 0; i < RPC; i++) {
        const int64_t ch = tid + i * TT;
        if (ch < D.nchunks) {
          T pp[W], sv[W], rr[W];
          ldc(D.p + ch * W, pp);
          ldc(D.s + ch * W, sv);
          ldc(D.g + ch * W, gv[i]);
          ldc(D.rT + ch * W, rr);
#pragma unroll
          for (int v = 0; v < W; v++) {
            sv[v] += T(alpha) * pp[v];
            gv[i][v] -= T(alpha) * yv[i][v];
            rs += double(rr[v]) * double(sv[v]);
            sg += double(sv[v]) * double(gv[i][v]);
            ss += double(sv[v]) * double(sv[v]);
          }
          stv(D.s + ch * W, sv);
          stv(D.g + ch * W, gv[i]);
          stv(D.z + ch * W, sent);
          stv(D.c0 + ch * W, sent);
        } else {
#pragma unroll
          for (int v = 0; v < W; v++) gv[i][v] = T(0);
        }
      }
      reset_queues(D);
      red_put(sh, 0, self_dot<T, RPC>(gv, gv));
      red_put(sh, 1, rs);
      red_put(sh, 2, sg);
      red_put(sh, 3, ss);
      dots_put<T, RPC>(sh, 4, D.S, D.npad, k, sh.order, D, gv, false);
      if (!reduce_all(D, sh, ctl, 4 + k, 33)) return false;
      tmark(sh, PH_UPDATE);
    }
    const double gn = sqrt(sh.sc[0]);
    const double rs = sh.sc[1], sg = sh.sc[2], ss = sh.sc[3];
    // Exit (iii), eq. "residual", without a product with A.  With x = u + s,
    // s orthogonal to Q (u is a column of Q), (A - theta I) u = r and
    // J s = -r - g, and neglecting v_i^T (A - theta I) s for the converged
    // v_i: ||A x - theta x||^2 = ||g||^2 + (r^T s)^2,
    // x^T (A - theta I) x = r^T s - s^T g, so rho - theta =
    // (r^T s - s^T g) / (1 + ||s||^2) and ||A x - rho x||^2 =
    // ||A x - theta x||^2 - (rho - theta)^2 (1 + ||s||^2).
    const double x2 = 1.0 + ss;
    const double dth = (rs - sg) / x2;
    const double e2 = gn * gn + rs * rs - dth * dth * x2;
    const double eres = sqrt(fmax(e2, 0.0) / x2);
    const double rho = theta + dth;
    res.gn = gn;
    res.eres = eres;
    res.rs = rs;
    if (gn <= O.tau_pcg * g0) {
      res.exit = 0;
      break;
    }
    if (O.exit_eigres && eres < O.tol * rho) {
      res.exit = 2;
      break;
    }
    if (O.exit_stag && l >= 1 && eres / eprev > gn / gprev) {
      res.exit = 3;
      break;
    }
    if (l + 1 == max_pcg) {
      res.exit = 1;
      break;
    }
    if (threadIdx.x == 0)
      for (int s = 0; s < k; s++) sh.sg[s] = sh.sc[4 + s];
    __syncthreads();
    gprev = gn;
    eprev = eres;
  }
  return true;
}

// ---------------------------------------------------------------------------
// FP64 pieces of the outer step
// ---------------------------------------------------------------------------

// Au = A u (FP64), returns u^T A u and u^T u in sh.sc[0..1].  u = Qt column j.
template <typename T, int RPC>
__device__ bool fp64_rayleigh(const Dev<T> &D, Shared &sh, Ctl &ctl, const double *u) {
  constexpr int W = VT<T>::W;
  const int64_t tid = gtid(), TT = gthreads();
  double uau = 0.0, uu = 0.0;
#pragma unroll
  for (int i = 0; i < RPC; i++) {
    const int64_t ch = tid + i * TT;
    if (ch < D.nchunks) {
      double acc[W], uv[W];
      sell_rows<W, double, double, double>(D.A64, u, ch, acc);
      ldc(u + ch * W, uv);
#pragma unroll
      for (int v = 0; v < W; v++) {
        uau += uv[v] * acc[v];
        uu += uv[v] * uv[v];
      }
      stv(D.Au + ch * W, acc);
    }
  }
  red_put(sh, 0, uau);
  red_put(sh, 1, uu);
  return reduce_all(D, sh, ctl, 2, 40);
}

// r = A u - theta u (FP64, and its working-precision copy rT), ||r||^2 in
// sh.sc[0]; shadows Q[:, j] = u.  With stage >= 0 (full BFGS update) the staged pair's second vector, which
// holds r_k, becomes w = r_k - r_{k+1} and sc[1] = s^T w.
template <typename T, int RPC>
__device__ bool fp64_residual(const Dev<T> &D, Shared &sh, Ctl &ctl, const double *u, double theta, int j,
                              int stage = -1) {
  constexpr int W = VT<T>::W;
  const int64_t tid = gtid(), TT = gthreads();
  double rr = 0.0, sw = 0.0;
  T *uq = D.Q + (int64_t)j * D.npad;
#pragma unroll
  for (int i = 0; i < RPC; i++) {
    const int64_t ch = tid + i * TT;
    if (ch < D.nchunks) {
      double au[W], uv[W], rv[W];
      ldc(D.Au + ch * W, au);
      ldc(u + ch * W, uv);
      T rt[W], ut[W];
#pragma unroll
      for (int v = 0; v < W; v++) {
        rv[v] = au[v] - theta * uv[v];
        rr += rv[v] * rv[v];
        rt[v] = T(rv[v]);
        ut[v] = T(uv[v]);
      }
      stv(D.r + ch * W, rv);
      stv(D.rT + ch * W, rt);
      stv(uq + ch * W, ut);
      if (stage >= 0) {
        T sv[W], wv[W];
        ldc(D.S + (int64_t)stage * D.npad + ch * W, sv);
        ldc(D.R + (int64_t)stage * D.npad + ch * W, wv);
#pragma unroll
        for (int v = 0; v < W; v++) {
          wv[v] = T(double(wv[v]) - rv[v]);
          sw += double(sv[v]) * double(wv[v]);
        }
        stv(D.R + (int64_t)stage * D.npad + ch * W, wv);
      }
    }
  }
  red_put(sh, 0, rr);
  if (stage >= 0) red_put(sh, 1, sw);
  return reduce_all(D, sh, ctl, stage >= 0 ? 2 : 1, 41);
}

template <typename T>
__device__ void load_state(const Dev<T> &D, Shared &sh, Ctl &ctl, const Opts &O, int gbase = 0, int gsize = -1) {
  if (threadIdx.x == 0) {
    s_gbase = gbase;
    s_gsize = gsize > 0 ? gsize : (int)gridDim.x;
  }
  ctl.epoch = 0;
  ctl.rbuf = 0;
  ctl.spin_ns = O.spin_ns;
  ctl.twarps = max(1, min(NWARP, O.trsv_warps));
  ctl.poll_ns = O.poll_ns;
  if (threadIdx.x == 0) {
    sh.ok = 1;
    for (int s = 0; s < KMAX; s++) sh.order[s] = s;
    for (int q = 0; q < 8; q++) sh.tacc[q] = 0;
    sh.tlast = gtimer();
  }
  __syncthreads();
}

// add this launch's phase times to the state (CTA 0)
__device__ __forceinline__ void flush_timers(State *st, Shared &sh) {
  if (lead_cta() && threadIdx.x == 0)
    for (int q = 0; q < 8; q++) st->tphase[q] += sh.tacc[q];
}

// ---------------------------------------------------------------------------
// Kernel: Newton iteration for eigenpair j (Algorithm 3.2, inner loop)
// ---------------------------------------------------------------------------
template <typename T, int RPC>
__device__ bool newton_body(const Dev<T> &D, const Opts &O, Shared &sh, Ctl &ctl, int j) {
  constexpr int W = VT<T>::W;
  const int64_t tid = gtid(), TT = gthreads();
  const int m = j + 1;
  double *u = D.Qt + (int64_t)j * D.npad;
  int k = 0;  // pairs reset for every eigenpair
  int spare = O.kmax;  // full update: physical slot staging the newest pair
  if (threadIdx.x == 0)
    for (int s = 0; s < KMAX; s++) sh.order[s] = s;
  __syncthreads();
  long long mvp = 0, pcg_total = 0, sum_m = 0, sum_k = 0;
  int pcg_sum = 0;
  int exits[5] = {0, 0, 0, 0, 0};

  if (!fp64_rayleigh<T, RPC>(D, sh, ctl, u)) return false;
  mvp++;
  double theta = sh.sc[0] / sh.sc[1];
  if (!fp64_residual<T, RPC>(D, sh, ctl, u, theta, j)) return false;
  double rnorm = sqrt(sh.sc[0]);
  tmark(sh, PH_OUTER);
  int it = 0;
  while (rnorm > O.tol * theta && it < O.max_newton) {
    if (!gram<T, RPC>(D, sh, ctl, m, k)) return false;
    tmark(sh, PH_OTHER);
    PcgOut po;
    if (!pcg_solve<T, RPC>(D, O, sh, ctl, m, k, theta, O.max_pcg, po)) return false;
    mvp += po.its;
    pcg_total += po.its;
    pcg_sum += po.its;
    sum_m += (long long)po.its * m;
    sum_k += (long long)po.its * k;
    exits[po.exit]++;
    // simplified update: store the pair (s_k, r_k) when alpha = s^T r_k < 0
    // (Theorem 3.2) in the ring of k_max slots.  Full update: copy (s_k, r_k)
    // into the spare slot; it becomes (s_k, r_k - r_{k+1}) with the next
    // residual and joins the ring if s^T w < 0.
    int slot = -1, stage = -1;
    if (O.kmax > 0 && O.bfgs_full) {
      stage = spare;
    } else if (O.kmax > 0 && po.rs < 0.0) {
      if (k < O.kmax) {
        slot = k;
        if (threadIdx.x == 0) sh.order[k] = k;
        k++;
      } else {
        if (threadIdx.x == 0) {
          slot = sh.order[0];
          for (int s = 0; s + 1 < k; s++) sh.order[s] = sh.order[s + 1];
          sh.order[k - 1] = slot;
        }
        __syncthreads();
        slot = sh.order[k - 1];
      }
    }
    __syncthreads();
    const int wslot = slot >= 0 ? slot : stage;
    // N1: t = u + s (FP64); copy the pair; ||t||^2, Qt^T t
    double tv[RPC][W];
    {
      double tt = 0.0;
#pragma unroll
      for (int i = 0; i < RPC; i++) {
        const int64_t ch = tid + i * TT;
        if (ch < D.nchunks) {
          double uv[W];
          T sv[W];
          ldc(u + ch * W, uv);
          ldc(D.s + ch * W, sv);
#pragma unroll
          for (int v = 0; v < W; v++) {
            tv[i][v] = uv[v] + double(sv[v]);
            tt += tv[i][v] * tv[i][v];
          }
          if (wslot >= 0) {
            T rt[W];
            ldc(D.rT + ch * W, rt);
            stv(D.S + (int64_t)wslot * D.npad + ch * W, sv);
            stv(D.R + (int64_t)wslot * D.npad + ch * W, rt);
          }
        } else {
#pragma unroll
          for (int v = 0; v < W; v++) tv[i][v] = 0.0;
        }
      }
      red_put(sh, 0, tt);
      for (int c = 0; c < j; c++) {
        const double *qc = D.Qt + (int64_t)c * D.npad;
        double acc = 0.0;
#pragma unroll
        for (int i = 0; i < RPC; i++) {
          const int64_t ch = tid + i * TT;
          if (ch < D.nchunks) {
            double q[W];
            ldc(qc + ch * W, q);
#pragma unroll
            for (int v = 0; v < W; v++) acc += q[v] * tv[i][v];
          }
        }
        red_put(sh, 1 + c, acc);
      }
      if (!reduce_all(D, sh, ctl, 1 + j, 42)) return false;
    }
    // N2: u = (t - Qt (Qt^T t)) / ||.||  (re-orthogonalisation against the
    // converged eigenvectors, then normalisation)
    {
      double nq = 0.0;
      for (int c = 0; c < j; c++) nq += sh.sc[1 + c] * sh.sc[1 + c];
      const double inv = 1.0 / sqrt(sh.sc[0] - nq);
      for (int c = 0; c < j; c++) {
        const double *qc = D.Qt + (int64_t)c * D.npad;
        const double cf = sh.sc[1 + c];
#pragma unroll
        for (int i = 0; i < RPC; i++) {
          const int64_t ch = tid + i * TT;
          if (ch < D.nchunks) {
            double q[W];
            ldc(qc + ch * W, q);
#pragma unroll
            for (int v = 0; v < W; v++) tv[i][v] -= cf * q[v];
          }
        }
      }
#pragma unroll
      for (int i = 0; i < RPC; i++) {
        const int64_t ch = tid + i * TT;
        if (ch < D.nchunks) {
#pragma unroll
          for (int v = 0; v < W; v++) tv[i][v] *= inv;
          stv(u + ch * W, tv[i]);
        }
      }
      if (!grid_sync(D.st, sh, ctl, 43)) return false;
    }
    if (!fp64_rayleigh<T, RPC>(D, sh, ctl, u)) return false;
    mvp++;
    theta = sh.sc[0] / sh.sc[1];
    if (!fp64_residual<T, RPC>(D, sh, ctl, u, theta, j, stage)) return false;
    rnorm = sqrt(sh.sc[0]);
    if (stage >= 0 && sh.sc[1] < 0.0) {
      // the staged pair joins the ring; the slot it replaces (or the lowest
      // free one) becomes the spare
      if (k < O.kmax) {
        if (threadIdx.x == 0) sh.order[k] = stage;
        k++;
        __syncthreads();
        for (spare = 0;; spare++) {
          bool used = false;
          for (int s = 0; s < k; s++) used = used || sh.order[s] == spare;
          if (!used) break;
        }
      } else {
        const int evicted = sh.order[0];
        __syncthreads();
        if (threadIdx.x == 0) {
          for (int s = 0; s + 1 < k; s++) sh.order[s] = sh.order[s + 1];
          sh.order[k - 1] = stage;
        }
        spare = evicted;
      }
      __syncthreads();
    }
    tmark(sh, PH_OUTER);
    it++;
  }
  flush_timers(D.st, sh);
  if (lead_cta() && threadIdx.x == 0) {
    State *st = D.st;
    st->theta = theta;
    st->rnorm = rnorm;
    st->lambda[j] = theta;
    st->res[j] = rnorm / theta;
    st->outer_its[j] = it;
    st->pcg_its[j] = pcg_sum;
    st->conv[j] = (rnorm <= O.tol * theta) ? 1 : 0;
    st->mvp_newton += mvp;
    st->pcg_total += pcg_total;
    st->pcg_sum_m += sum_m;
    st->pcg_sum_k += sum_k;
    for (int e = 0; e < 5; e++) st->exits[e] += exits[e];
  }
  return true;
}

template <typename T, int RPC, int CH>
__global__ void __launch_bounds__(TPB, 1) k_newton(Dev<T> D, Opts O) {
  __shared__ Shared sh;
  Ctl ctl;
  load_state(D, sh, ctl, O);
  newton_body<T, RPC>(D, O, sh, ctl, D.st->j);
}

// ---------------------------------------------------------------------------
// Kernel: DACG for eigenpair j (Section 4.1): preconditioned nonlinear CG on
// the Rayleigh quotient in the complement of the converged eigenvectors.
// On entry x holds the start vector; on exit Qt[:, j] holds u_0 (FP64).
// ---------------------------------------------------------------------------
template <typename T, int RPC>
__device__ bool dacg_body(const Dev<T> &D, const Opts &O, Shared &sh, Ctl &ctl, int j) {
  constexpr int W = VT<T>::W;
  const int64_t tid = gtid(), TT = gthreads();
  const int mq = j;  // converged eigenvectors (shadow columns of Q)
  const T Tsent = sentinel<T>();
  long long mvp = 0;
  T xv[RPC][W];
#pragma unroll
  for (int i = 0; i < RPC; i++) {
    const int64_t ch = tid + i * TT;
    if (ch < D.nchunks)
      ldc((D.X0 ? D.X0 + (int64_t)j * D.npad : D.x) + ch * W, xv[i]);
    else
#pragma unroll
      for (int v = 0; v < W; v++) xv[i][v] = T(0);
  }
  // x0 projected on the complement of Q~ twice (classical Gram-Schmidt)
  for (int rep = 0; rep < 2 && mq > 0; rep++) {
    dots_put<T, RPC>(sh, 0, D.Q, D.npad, mq, nullptr, D, xv, false);
    if (!reduce_all(D, sh, ctl, mq, 50)) return false;
    for (int c = threadIdx.x; c < mq; c += TPB) sh.qv[c] = -sh.sc[c];
    __syncthreads();
    comb_add<T, RPC>(D.Q, D.npad, mq, sh.qv, nullptr, D, xv, 1.0);
  }
  red_put(sh, 0, self_dot<T, RPC>(xv, xv));
  if (!reduce_all(D, sh, ctl, 1, 51)) return false;
  {
    const T inv = T(1.0 / sqrt(sh.sc[0]));
#pragma unroll
    for (int i = 0; i < RPC; i++) {
      const int64_t ch = tid + i * TT;
#pragma unroll
      for (int v = 0; v < W; v++) xv[i][v] *= inv;
      if (ch < D.nchunks) stv(D.x + ch * W, xv[i]);
    }
  }
  if (!grid_sync(D.st, sh, ctl, 52)) return false;
  // Ax
#pragma unroll
  for (int i = 0; i < RPC; i++) {
    const int64_t ch = tid + i * TT;
    if (ch < D.nchunks) {
      T acc[W];
      sell_rows<W, T, T, T>(D.A, D.x, ch, acc);
      stv(D.Ax + ch * W, acc);
    }
  }
  mvp++;
  if (!grid_sync(D.st, sh, ctl, 53)) return false;

  double nx = 1.0, gg_prev = 0.0;
  int its = 0;
  for (int it = 0; it < O.max_dacg; it++) {
    // P1: normalise x, Ax by the last norm; q = x^T A x, f = x^T x
    T av[RPC][W];
    {
      const T inv = T(1.0 / nx);
#pragma unroll
      for (int i = 0; i < RPC; i++) {
        const int64_t ch = tid + i * TT;
        if (ch < D.nchunks) {
          ldc(D.x + ch * W, xv[i]);
          ldc(D.Ax + ch * W, av[i]);
          if (nx != 1.0) {
#pragma unroll
            for (int v = 0; v < W; v++) xv[i][v] *= inv, av[i][v] *= inv;
            stv(D.x + ch * W, xv[i]);
            stv(D.Ax + ch * W, av[i]);
          }
        } else {
#pragma unroll
          for (int v = 0; v < W; v++) xv[i][v] = T(0), av[i][v] = T(0);
        }
      }
      red_put(sh, 0, self_dot<T, RPC>(xv, av));
      red_put(sh, 1, self_dot<T, RPC>(xv, xv));
      if (!reduce_all(D, sh, ctl, 2, 54)) return false;
      nx = 1.0;  // x and Ax now hold the normalised iterate
    }
    const double q = sh.sc[0], f = sh.sc[1];
    // P2: g = A x - q x, ||g||; reset the solve outputs
    T gv[RPC][W];
    {
      T sent[W];
#pragma unroll
      for (int v = 0; v < W; v++) sent[v] = Tsent;
#pragma unroll
      for (int i = 0; i < RPC; i++) {
        const int64_t ch = tid + i * TT;
#pragma unroll
        for (int v = 0; v < W; v++) gv[i][v] = av[i][v] - T(q) * xv[i][v];
        if (ch < D.nchunks) {
          stv(D.g + ch * W, gv[i]);
          stv(D.z + ch * W, sent);
          stv(D.c0 + ch * W, sent);
        }
      }
      reset_queues(D);
      red_put(sh, 0, self_dot<T, RPC>(gv, gv));
      if (!reduce_all(D, sh, ctl, 1, 55)) return false;
      tmark(sh, PH_UPDATE);
    }
    if (sqrt(sh.sc[0]) <= O.tau_dacg * q) break;
    // P3-P5: gt = (I - Q~Q~^T) Phat_0 g,  p = -gt + beta p
    double gg;
    {
      // Phat_0 g via the preconditioner tail with no pairs, writing into Ap as
      // scratch: Ap = c0 - Q z, then p = -Ap + beta p below.
      if (!precond_tail<T, RPC>(D, sh, ctl, mq, 0, D.Ap, 0.0, false, &gg)) return false;
      const double beta = (it == 0) ? 0.0 : gg / gg_prev;
#pragma unroll
      for (int i = 0; i < RPC; i++) {
        const int64_t ch = tid + i * TT;
        if (ch < D.nchunks) {
          T gt[W], pp[W];
          ldc(D.Ap + ch * W, gt);
          if (it > 0) {
            ldc(D.p + ch * W, pp);
#pragma unroll
            for (int v = 0; v < W; v++) pp[v] = -gt[v] + T(beta) * pp[v];
          } else {
#pragma unroll
            for (int v = 0; v < W; v++) pp[v] = -gt[v];
          }
          stv(D.p + ch * W, pp);
        }
      }
      if (!grid_sync(D.st, sh, ctl, 56)) return false;
      tmark(sh, PH_DIR);
    }
    // P6: Ap = A p; line-search scalars
    {
      double a = 0.0, b = 0.0, d = 0.0, e = 0.0;
#pragma unroll
      for (int i = 0; i < RPC; i++) {
        const int64_t ch = tid + i * TT;
        if (ch < D.nchunks) {
          T acc[W], pp[W];
          sell_rows<W, T, T, T>(D.A, D.p, ch, acc);
          ldc(D.p + ch * W, pp);
#pragma unroll
          for (int v = 0; v < W; v++) {
            a += double(pp[v]) * double(acc[v]);
            b += double(xv[i][v]) * double(acc[v]);
            d += double(pp[v]) * double(pp[v]);
            e += double(xv[i][v]) * double(pp[v]);
          }
          stv(D.Ap + ch * W, acc);
        }
      }
      mvp++;
      red_put(sh, 0, a);
      red_put(sh, 1, b);
      red_put(sh, 2, d);
      red_put(sh, 3, e);
      if (!reduce_all(D, sh, ctl, 4, 57)) return false;
      tmark(sh, PH_SPMV);
    }
    double al;
    {
      const double a = sh.sc[0], b = sh.sc[1], c = q, d = sh.sc[2], e = sh.sc[3];
      const double A2 = a * e - b * d, B2 = a * f - c * d, C2 = b * f - c * e;
      if (A2 == 0.0) {
        al = (B2 != 0.0) ? -C2 / B2 : 0.0;
      } else {
        const double disc = fmax(B2 * B2 - 4.0 * A2 * C2, 0.0);
        const double t = -0.5 * (B2 + copysign(sqrt(disc), B2));
        const double r1 = t / A2;
        al = r1;
        if (t != 0.0) {
          const double r2 = C2 / t;
          const double q1 = (c + 2 * r1 * b + r1 * r1 * a) / (f + 2 * r1 * e + r1 * r1 * d);
          const double q2 = (c + 2 * r2 * b + r2 * r2 * a) / (f + 2 * r2 * e + r2 * r2 * d);
          if (q2 < q1) al = r2;
        }
      }
    }
    // P7: x += al p, Ax += al Ap, ||x||
    {
      double xx = 0.0;
#pragma unroll
      for (int i = 0; i < RPC; i++) {
        const int64_t ch = tid + i * TT;
        if (ch < D.nchunks) {
          T pp[W], ap[W];
          ldc(D.p + ch * W, pp);
          ldc(D.Ap + ch * W, ap);
#pragma unroll
          for (int v = 0; v < W; v++) {
            xv[i][v] += T(al) * pp[v];
            av[i][v] += T(al) * ap[v];
            xx += double(xv[i][v]) * double(xv[i][v]);
          }
          stv(D.x + ch * W, xv[i]);
          stv(D.Ax + ch * W, av[i]);
        }
      }
      red_put(sh, 0, xx);
      if (!reduce_all(D, sh, ctl, 1, 58)) return false;
      nx = sqrt(sh.sc[0]);
      tmark(sh, PH_UPDATE);
    }
    its = it + 1;
    if (O.recompute > 0 && its % O.recompute == 0) {
#pragma unroll
      for (int i = 0; i < RPC; i++) {
        const int64_t ch = tid + i * TT;
        if (ch < D.nchunks) {
          T acc[W];
          sell_rows<W, T, T, T>(D.A, D.x, ch, acc);
          stv(D.Ax + ch * W, acc);
        }
      }
      mvp++;
      if (!grid_sync(D.st, sh, ctl, 59)) return false;
    }
    gg_prev = gg;
  }
  // u_0 = x / ||x|| in FP64 into Qt[:, j]
  {
    double *u = D.Qt + (int64_t)j * D.npad;
#pragma unroll
    for (int i = 0; i < RPC; i++) {
      const int64_t ch = tid + i * TT;
      if (ch < D.nchunks) {
        T xx[W];
        ldc(D.x + ch * W, xx);
        double uv[W];
#pragma unroll
        for (int v = 0; v < W; v++) uv[v] = double(xx[v]) / nx;
        stv(u + ch * W, uv);
      }
    }
  }
  flush_timers(D.st, sh);
  if (lead_cta() && threadIdx.x == 0) {
    D.st->dacg_its[j] = its;
    D.st->mvp_dacg += mvp;
    D.st->dacg_total += its;
    D.st->dacg_sum_m += (long long)its * mq;
  }
  return true;
}

template <typename T, int RPC, int CH>
__global__ void __launch_bounds__(TPB, 1) k_dacg(Dev<T> D, Opts O) {
  __shared__ Shared sh;
  Ctl ctl;
  load_state(D, sh, ctl, O);
  dacg_body<T, RPC>(D, O, sh, ctl, D.st->j);
}

// ---------------------------------------------------------------------------
// Kernels exposing single building blocks (verification entry points)
// ---------------------------------------------------------------------------

// y = (A - theta I) x  (x in D.p, y in D.y)
template <typename T, int RPC, int CH>
__global__ void __launch_bounds__(TPB, 1) k_shifted(Dev<T> D, double theta) {
  constexpr int W = VT<T>::W;
  if (threadIdx.x == 0) {
    s_gbase = 0;
    s_gsize = (int)gridDim.x;
  }
  __syncthreads();
  const int64_t tid = gtid(), TT = gthreads();
#pragma unroll
  for (int i = 0; i < RPC; i++) {
    const int64_t ch = tid + i * TT;
    if (ch < D.nchunks) {
      T acc[W], pp[W];
      sell_rows<W, T, T, T>(D.A, D.p, ch, acc);
      ldc(D.p + ch * W, pp);
#pragma unroll
      for (int v = 0; v < W; v++) acc[v] -= T(theta) * pp[v];
      stv(D.y + ch * W, acc);
    }
  }
}

// c = P_k g by Algorithm 3.1 (g in D.g, output in D.y); m columns of Q, k pairs
// in slots 0..k-1 (chronological).
template <typename T, int RPC, int CH>
__global__ void __launch_bounds__(TPB, 1) k_prec(Dev<T> D, Opts O, int m, int k) {
  constexpr int W = VT<T>::W;
  __shared__ Shared sh;
  Ctl ctl;
  load_state(D, sh, ctl, O);
  if (threadIdx.x == 0)
    for (int s = 0; s < KMAX; s++) sh.order[s] = s;
  __syncthreads();
  if (!gram<T, RPC>(D, sh, ctl, m, k)) return;
  const int64_t tid = gtid(), TT = gthreads();
  const T Tsent = sentinel<T>();
  T gv[RPC][W];
  T sent[W];
#pragma unroll
  for (int v = 0; v < W; v++) sent[v] = Tsent;
#pragma unroll
  for (int i = 0; i < RPC; i++) {
    const int64_t ch = tid + i * TT;
    if (ch < D.nchunks) {
      ldc(D.g + ch * W, gv[i]);
      stv(D.z + ch * W, sent);
      stv(D.c0 + ch * W, sent);
    } else {
#pragma unroll
      for (int v = 0; v < W; v++) gv[i][v] = T(0);
    }
  }
  reset_queues(D);
  dots_put<T, RPC>(sh, 0, D.S, D.npad, k, sh.order, D, gv, false);
  if (!reduce_all(D, sh, ctl, k, 60)) return;
  if (threadIdx.x == 0)
    for (int s = 0; s < k; s++) sh.sg[s] = sh.sc[s];
  __syncthreads();
  coef_a(sh, k);
  double gamma;
  precond_tail<T, RPC>(D, sh, ctl, m, k, D.y, 0.0, false, &gamma);
}

// One inner solve: theta given, r in rT, Q with m columns, k pairs in slots 0..k-1.
template <typename T, int RPC, int CH>
__global__ void __launch_bounds__(TPB, 1) k_pcg(Dev<T> D, Opts O, int m, int k, double theta, int max_pcg) {
  __shared__ Shared sh;
  Ctl ctl;
  load_state(D, sh, ctl, O);
  if (threadIdx.x == 0)
    for (int s = 0; s < KMAX; s++) sh.order[s] = s;
  __syncthreads();
  if (!gram<T, RPC>(D, sh, ctl, m, k)) return;
  PcgOut po;
  if (!pcg_solve<T, RPC>(D, O, sh, ctl, m, k, theta, max_pcg, po)) return;
  if (lead_cta() && threadIdx.x == 0) {
    D.st->last_its = po.its;
    D.st->last_exit = po.exit;
    D.st->last_g0 = po.g0;
    D.st->last_gn = po.gn;
    D.st->last_eres = po.eres;
  }
}

// ---------------------------------------------------------------------------
// Kernel: adjoint solve for eigenvector j (not in the paper).
// On entry b64 holds gbar_j (device order, FP64, already multiplied by the
// sign of the output eigenvector); Qt holds v_1..v_p (FP64) and Q their
// working-precision shadows; st->lambda the eigenvalues.  Computes
//   c_i = v_i^T gbar,   b = gbar - V c,
//   y perp V solving (I-VV^T)(A - lambda_j I)(I-VV^T) y = b,
//   xi = -sum_{i != j} v_i c_i / (lambda_i - lambda_j) - y   (written to t),
// the solve by iterative refinement: FP64 residual rho = b - (I-VV^T)(A -
// lambda_j I) y with the FP64 matrix, correction by the inner projected PCG
// of the correction equation (Q = V, IC preconditioner, shift lambda_j) in the
// working precision, until ||rho|| <= tol ||b||.
// ---------------------------------------------------------------------------
template <typename T, int RPC>
__device__ bool fp64_project_dots(const Dev<T> &D, Shared &sh, Ctl &ctl, int p, const double (&v)[RPC][VT<T>::W],
                                  int where) {
  constexpr int W = VT<T>::W;
  const int64_t tid = gtid(), TT = gthreads();
  int c = 0;
  for (; c < p; c++) {
    const double *qc = D.Qt + (int64_t)c * D.npad;
    double acc = 0.0;
#pragma unroll
    for (int i = 0; i < RPC; i++) {
      const int64_t ch = tid + i * TT;
      if (ch < D.nchunks) {
        double q[W];
        ldc(qc + ch * W, q);
#pragma unroll
        for (int u = 0; u < W; u++) acc += q[u] * v[i][u];
      }
    }
    red_put(sh, c, acc);
  }
  return reduce_all(D, sh, ctl, p, where);
}

template <typename T, int RPC>
__device__ void fp64_comb_add(const Dev<T> &D, int p, const double *coef, double sgn, double (&v)[RPC][VT<T>::W]) {
  constexpr int W = VT<T>::W;
  const int64_t tid = gtid(), TT = gthreads();
  for (int c = 0; c < p; c++) {
    const double *qc = D.Qt + (int64_t)c * D.npad;
    const double cf = sgn * coef[c];
#pragma unroll
    for (int i = 0; i < RPC; i++) {
      const int64_t ch = tid + i * TT;
      if (ch < D.nchunks) {
        double q[W];
        ldc(qc + ch * W, q);
#pragma unroll
        for (int u = 0; u < W; u++) v[i][u] += cf * q[u];
      }
    }
  }
}

template <typename T, int RPC, int CH>
__global__ void __launch_bounds__(TPB, 1) k_adjoint(Dev<T> D, Opts O, int j, int p, double tol, int max_refine) {
  constexpr int W = VT<T>::W;
  __shared__ Shared sh;
  Ctl ctl;
  load_state(D, sh, ctl, O);
  const int64_t tid = gtid(), TT = gthreads();
  const double lam = D.st->lambda[j];
  double v[RPC][W];
  // 1-2: c = V^T gbar, b = gbar - V c, y = 0
#pragma unroll
  for (int i = 0; i < RPC; i++) {
    const int64_t ch = tid + i * TT;
    if (ch < D.nchunks)
      ldc(D.b64 + ch * W, v[i]);
    else
#pragma unroll
      for (int u = 0; u < W; u++) v[i][u] = 0.0;
  }
  if (!fp64_project_dots<T, RPC>(D, sh, ctl, p, v, 70)) return;
  for (int c = threadIdx.x; c < p; c += TPB) sh.cadj[c] = sh.sc[c];
  __syncthreads();
  fp64_comb_add<T, RPC>(D, p, sh.cadj, -1.0, v);
  {
    double bb = 0.0;
    const double zero[W] = {};
#pragma unroll
    for (int i = 0; i < RPC; i++) {
      const int64_t ch = tid + i * TT;
      if (ch < D.nchunks) {
        stv(D.b64 + ch * W, v[i]);
        double zz[W];
#pragma unroll
        for (int u = 0; u < W; u++) zz[u] = zero[u];
        stv(D.y64 + ch * W, zz);
#pragma unroll
        for (int u = 0; u < W; u++) bb += v[i][u] * v[i][u];
      }
    }
    red_put(sh, 0, bb);
    if (!reduce_all(D, sh, ctl, 1, 71)) return;
  }
  const double bn = sqrt(sh.sc[0]);
  int refine = 0, inner = 0;
  double res = 0.0;
  for (int it = 0; bn > 0.0 && it < max_refine; it++) {
    // a: w = (A - lambda I) y in FP64, V^T w
    double w[RPC][W];
#pragma unroll
    for (int i = 0; i < RPC; i++) {
      const int64_t ch = tid + i * TT;
      if (ch < D.nchunks) {
        double acc[W], yy[W];
        sell_rows<W, double, double, double>(D.A64, D.y64, ch, acc);
        ldc(D.y64 + ch * W, yy);
#pragma unroll
        for (int u = 0; u < W; u++) w[i][u] = acc[u] - lam * yy[u];
      } else {
#pragma unroll
        for (int u = 0; u < W; u++) w[i][u] = 0.0;
      }
    }
    if (!fp64_project_dots<T, RPC>(D, sh, ctl, p, w, 72)) return;
    for (int c = threadIdx.x; c < p; c += TPB) sh.qv[c] = sh.sc[c];
    __syncthreads();
    fp64_comb_add<T, RPC>(D, p, sh.qv, -1.0, w);  // w = (I - VV^T)(A - lambda I) y
    // b: rho = b - w, ||rho||, rT = -rho
    {
      double rr = 0.0;
#pragma unroll
      for (int i = 0; i < RPC; i++) {
        const int64_t ch = tid + i * TT;
        if (ch < D.nchunks) {
          double bv[W];
          T rt[W];
          ldc(D.b64 + ch * W, bv);
#pragma unroll
          for (int u = 0; u < W; u++) {
            const double rho = bv[u] - w[i][u];
            rr += rho * rho;
            rt[u] = T(-rho);
          }
          stv(D.rT + ch * W, rt);
        }
      }
      red_put(sh, 0, rr);
      if (!reduce_all(D, sh, ctl, 1, 73)) return;
    }
    res = sqrt(sh.sc[0]) / bn;
    if (res <= tol) break;
    // d: correction by the inner projected PCG (J s = rho)
    PcgOut po;
    if (!pcg_solve<T, RPC>(D, O, sh, ctl, p, 0, lam, O.max_pcg, po)) return;
    inner += po.its;
    refine++;
    // e: y += s, then y -= V V^T y
    double yv[RPC][W];
#pragma unroll
    for (int i = 0; i < RPC; i++) {
      const int64_t ch = tid + i * TT;
      if (ch < D.nchunks) {
        T sv[W];
        ldc(D.y64 + ch * W, yv[i]);
        ldc(D.s + ch * W, sv);
#pragma unroll
        for (int u = 0; u < W; u++) yv[i][u] += double(sv[u]);
      } else {
#pragma unroll
        for (int u = 0; u < W; u++) yv[i][u] = 0.0;
      }
    }
    if (!fp64_project_dots<T, RPC>(D, sh, ctl, p, yv, 74)) return;
    for (int c = threadIdx.x; c < p; c += TPB) sh.qv[c] = sh.sc[c];
    __syncthreads();
    fp64_comb_add<T, RPC>(D, p, sh.qv, -1.0, yv);
#pragma unroll
    for (int i = 0; i < RPC; i++) {
      const int64_t ch = tid + i * TT;
      if (ch < D.nchunks) stv(D.y64 + ch * W, yv[i]);
    }
    if (!grid_sync(D.st, sh, ctl, 75)) return;
  }
  // xi = -y - sum_{i != j} v_i c_i / (lambda_i - lambda_j)
  if (threadIdx.x == 0)
    for (int c = 0; c < p; c++) sh.qv[c] = (c == j) ? 0.0 : sh.cadj[c] / (D.st->lambda[c] - lam);
  __syncthreads();
  {
    double xi[RPC][W];
#pragma unroll
    for (int i = 0; i < RPC; i++) {
      const int64_t ch = tid + i * TT;
      if (ch < D.nchunks) {
        ldc(D.y64 + ch * W, xi[i]);
#pragma unroll
        for (int u = 0; u < W; u++) xi[i][u] = -xi[i][u];
      } else {
#pragma unroll
        for (int u = 0; u < W; u++) xi[i][u] = 0.0;
      }
    }
    fp64_comb_add<T, RPC>(D, p, sh.qv, -1.0, xi);
#pragma unroll
    for (int i = 0; i < RPC; i++) {
      const int64_t ch = tid + i * TT;
      if (ch < D.nchunks) stv(D.t + ch * W, xi[i]);
    }
  }
  if (lead_cta() && threadIdx.x == 0) {
    D.st->adj_refine = refine;
    D.st->adj_inner = inner;
    D.st->adj_res = res;
  }
}

// ---------------------------------------------------------------------------
// Kernel: batched solve.  Groups of B.G consecutive CTAs take problems from a
// device work queue (largest first); a group runs the whole of Algorithm 3.2
// for its problem (DACG and Newton for every eigenpair) with group-relative
// barriers and reductions, then takes the next problem.  A problem whose
// layout was built for g < G CTAs runs on the first g CTAs of the group.
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ bool group_sync(const Batch<T> &B, int group, unsigned &gepoch, Shared &sh) {
  __syncthreads();
  if (threadIdx.x == 0) {
    gepoch++;
    const unsigned target = gepoch * (unsigned)B.G;
    __threadfence();
    red_release_add(&B.gbar[group], 1u);
    long long t0 = 0;
    int spins = 0;
    int ok = 1;
    while (ld_acquire(&B.gbar[group]) < target) {
      if (++spins >= 64) {
        spins = 0;
        __nanosleep(256);
        if (ld_relaxed_int(&B.gerr[group]) != 0) {
          ok = 0;
          break;
        }
        const long long now = gtimer();
        if (t0 == 0)
          t0 = now;
        else if (now - t0 > B.group_spin_ns) {
          atomicExch(&B.gerr[group], 8 /*NLE_ERR_TIMEOUT*/);
          ok = 0;
          break;
        }
      }
    }
    __threadfence();
    sh.ok = ok && ld_relaxed_int(&B.gerr[group]) == 0;
  }
  __syncthreads();
  return sh.ok != 0;
}

template <typename T, int RPC, int CH>
__global__ void __launch_bounds__(TPB, 1) k_batch(Batch<T> B, Opts O) {
  __shared__ Shared sh;
  __shared__ __align__(16) unsigned char sD_raw[sizeof(Dev<T>)];  // problem descriptor
  Dev<T> &sD = *reinterpret_cast<Dev<T> *>(sD_raw);
  __shared__ int s_idx;
  const int group = (int)blockIdx.x / B.G, rank = (int)blockIdx.x % B.G;
  unsigned gepoch = 0;
  for (;;) {
    if (rank == 0 && threadIdx.x == 0) {
      const unsigned idx = atomicAdd(B.queue, 1u);
      atomicExch(&B.gslot[group], (int)idx);
    }
    if (!group_sync(B, group, gepoch, sh)) return;
    if (threadIdx.x == 0) s_idx = ld_relaxed_int(&B.gslot[group]);
    __syncthreads();
    const int idx = s_idx;
    if (idx >= B.count) return;
    if (threadIdx.x == 0) sD = B.devs[B.order[idx]];
    __syncthreads();
    const int gi = sD.grid;
    if (rank < gi) {
      Ctl ctl;
      load_state(sD, sh, ctl, O, group * B.G, gi);
      for (int j = 0; j < B.p; j++) {
        if (!dacg_body<T, RPC>(sD, O, sh, ctl, j)) break;
        if (!grid_sync(sD.st, sh, ctl, 80)) break;
        if (!newton_body<T, RPC>(sD, O, sh, ctl, j)) break;
        if (!grid_sync(sD.st, sh, ctl, 81)) break;
      }
    }
    // every CTA of the group is done with this problem before the slot moves on
    if (!group_sync(B, group, gepoch, sh)) return;
  }
}

// ---------------------------------------------------------------------------
// host-side launch table.  This file is compiled once per (precision, RPC,
// triangular solves) triple (NLE_T, NLE_RPC, NLE_TRSV_TU, NLE_TAG defined by the build) so that the
// instantiations compile in parallel.
// ---------------------------------------------------------------------------
#if defined(NLE_T) && defined(NLE_RPC) && defined(NLE_TAG)
#define NLE_CAT2(a, b) a##b
#define NLE_CAT(a, b) NLE_CAT2(a, b)
void *NLE_CAT(kernel_ptr_, NLE_TAG)(int id) {
  switch (id) {
    case 0: return (void *)k_newton<NLE_T, NLE_RPC, NLE_TRSV_TU>;
    case 1: return (void *)k_dacg<NLE_T, NLE_RPC, NLE_TRSV_TU>;
    case 2: return (void *)k_shifted<NLE_T, NLE_RPC, NLE_TRSV_TU>;
    case 3: return (void *)k_prec<NLE_T, NLE_RPC, NLE_TRSV_TU>;
    case 4: return (void *)k_pcg<NLE_T, NLE_RPC, NLE_TRSV_TU>;
    case 5: return (void *)k_adjoint<NLE_T, NLE_RPC, NLE_TRSV_TU>;
    case 6: return (void *)k_batch<NLE_T, NLE_RPC, NLE_TRSV_TU>;
  }
  return nullptr;
}
#endif

}  // namespace nle
