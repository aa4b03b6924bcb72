// Host-only test shim: the steps of the triangular solves (plan_steps,
// build_steps of nle_setup.cpp) without a GPU, for tests/test_steps_layout.py.
// Built by that test with g++; not part of the library.
#include <cstring>
#include <vector>

#include "../paper_1312_1553_gb300/csrc/nle_internal.h"
#include "../paper_1312_1553_gb300/csrc/nle_setup.h"

using namespace nle;

static StepsHost<double> g_S64;
static StepsHost<float> g_S32;
static std::vector<int32_t> g_perm;
static std::vector<double> g_diag;

template <typename T>
static void fill(const Permuted &P, int64_t rows, bool lower, int lpr, int nwarps, StepsHost<T> &S, int64_t *sizes) {
  plan_steps<T>(P, rows, lower, lpr, nwarps, S);
  build_steps<T>(P, rows, lower, lpr, S);
  sizes[1] = (int64_t)S.hptr.size() - 1;
  sizes[2] = (int64_t)S.head.size();
  sizes[3] = (int64_t)S.opnd.size();
  sizes[4] = (int64_t)S.hpos.size();
  sizes[5] = S.halo_max;
}

// colors: 0 natural ordering, 1 or 2 the multicolour ordering of that distance;
// dbl: FP64, else FP32; solve slabs of m slabs of bsize rows.  sizes: npad,
// solve slabs, steps, entries, halo values, halo_max.
extern "C" int shim_steps(int64_t n, const int64_t *rp, const int32_t *ci, const double *va, int lfil, double tau,
                          int colors, int lower, int dbl, int64_t bsize, int m, int lpr, int nwarps, int64_t *sizes) {
  std::vector<int32_t> P0;
  std::vector<int64_t> brp;
  std::vector<int32_t> bci;
  std::vector<double> bva;
  if (colors) {
    multicolor_order(n, rp, ci, colors, P0);
    permute_csr(n, rp, ci, va, P0, brp, bci, bva);
    rp = brp.data(), ci = bci.data(), va = bva.data();
  }
  Factor F;
  int64_t bad = -1;
  if (ic_factor_host(n, rp, ci, va, lfil, tau, F, &bad) != 0) return -1;
  const int64_t npad = (n + 127) / 128 * 128;
  std::vector<int32_t> iperm;
  slab_level_order(F, bsize, P0.empty() ? nullptr : P0.data(), g_perm, iperm);
  Permuted P;
  permute(n, rp, ci, va, F, g_perm, iperm, npad, P);
  g_diag = P.diag;
  if (dbl) fill<double>(P, m * bsize, lower != 0, lpr, nwarps, g_S64, sizes);
  else fill<float>(P, m * bsize, lower != 0, lpr, nwarps, g_S32, sizes);
  if (colors)
    for (int64_t i = 0; i < n; i++) g_perm[i] = P0[g_perm[i]];
  sizes[0] = npad;
  return 0;
}

template <typename T>
static void get(const StepsHost<T> &S, int32_t *step0, int32_t *head, int32_t *row, int32_t *opnd, double *val,
                int32_t *hptr, int32_t *hpos) {
  memcpy(step0, S.step0.data(), S.step0.size() * 4);
  memcpy(head, S.head.data(), S.head.size() * sizeof(StepHead));
  memcpy(row, S.row.data(), S.row.size() * 4);
  memcpy(opnd, S.opnd.data(), S.opnd.size() * 4);
  for (size_t i = 0; i < S.val.size(); i++) val[i] = S.val[i];
  memcpy(hptr, S.hptr.data(), S.hptr.size() * 4);
  memcpy(hpos, S.hpos.data(), S.hpos.size() * 4);
}

extern "C" void shim_steps_get(int dbl, int32_t *step0, int32_t *head, int32_t *row, int32_t *opnd, double *val,
                               int32_t *hptr, int32_t *hpos, double *diag, int32_t *perm) {
  if (dbl) get(g_S64, step0, head, row, opnd, val, hptr, hpos);
  else get(g_S32, step0, head, row, opnd, val, hptr, hpos);
  memcpy(diag, g_diag.data(), g_diag.size() * 8);
  memcpy(perm, g_perm.data(), g_perm.size() * 4);
}
