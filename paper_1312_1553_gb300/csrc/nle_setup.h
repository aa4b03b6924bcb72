// Host-side set-up of the nle library (see nle_setup.cpp).
#pragma once
#include <cstdint>
#include <string>
#include <future>
#include <system_error>
#include <vector>

#include "nle_internal.h"

namespace nle {

struct Factor {
  int64_t n = 0;
  // L by rows, diagonal last (exported by nle_get_factor)
  std::vector<int64_t> Lrowptr;
  std::vector<int32_t> Lcol;
  std::vector<double> Lval;
  // L by columns, diagonal first (= U = L^T by rows)
  std::vector<int64_t> Ccolptr;
  std::vector<int32_t> Crow;
  std::vector<double> Cval;
  std::vector<int32_t> levL, levU;
  int64_t nlevL = 0, nlevU = 0;
};

// Relabelled (slab-major, level-minor) matrices, row by row.
struct Permuted {
  int64_t n = 0, npad = 0;
  std::vector<int64_t> Arp, Lrp, Urp;
  std::vector<int32_t> Acol, Lcol, Ucol;
  std::vector<double> Aval, Lval, Uval, diag;
  std::vector<int32_t> lev;   // level (of L) of every relabelled row
  std::vector<int32_t> levU;  // level (of U = L^T) of every relabelled row
};

template <typename TV>
struct SellHost {
  int64_t nslices = 0;
  std::vector<int64_t> sptr;
  std::vector<int32_t> col;
  std::vector<TV> val;
};

// Strictly triangular part in per-slab ELL form (see trsv_block).
template <typename TV>
struct EllHost {
  std::vector<int64_t> off;    // per slab: first entry
  std::vector<int32_t> width;  // per slab: entries per row, multiple of 8
  std::vector<int32_t> col;    // -1 = padding
  std::vector<TV> val;
  // per row (level schedule): bits 0-3 its round inside its group of R
  // rows, bits 4-7 the group's last round, bits 8-15 the group's overflow
  // steps (entries past the 2 * 32 / R a warp step prefetches, in steps of
  // 32 / R; 255: up to the slab's width)
  std::vector<uint16_t> round;
};

// Steps of one strictly triangular factor.  The rows of each solve slab (some
// consecutive slabs) are sorted by level, then position (the other way round
// for L^T), and cut at every change of level and after every 32 / lpr rows (lpr
// lanes per row).  An operand is the offset of its value in the solve slab's
// shared-memory window: its own results, a slot that holds 0, and its halo
// (the values of other solve slabs, in the order in which the steps first
// need them).
// Entry k of a row belongs to lane k % lpr of the row and is that lane's entry
// number k / lpr; a lane's entries come in quads of four, padded with zeros,
// and a step stores quad after quad, lane after lane.
// Steps that follow each other belong to consecutive ones of nwarps warps.
// Where the warps of two consecutive levels are all different, every step of
// the second starts with a barrier of its warp and of all warps of the first.
// Elsewhere the first step of a level starts with a barrier of its warp and
// of all warps of the level before (of that level's last step only, with
// STEP_WAIT, if these are too many), and each step releases the next one of
// its level (STEP_EARLY).
template <typename TV>
struct StepsHost {
  std::vector<int32_t> step0;  // per solve slab + 1: first step
  std::vector<StepHead> head;  // per step
  std::vector<int32_t> row;    // 32 / lpr per step: rows, relative to the solve slab
  std::vector<int32_t> opnd;   // operands, in bytes from the start of the CTA's dynamic shared memory
  std::vector<TV> val;         // coefficients, same order
  std::vector<int32_t> hptr;   // per solve slab + 1: first halo value
  std::vector<int32_t> hpos;   // position of every halo value
  int64_t halo_max = 0;        // largest halo of a solve slab
  int n_max = 0;               // most entries of a lane
  bool fits = false;           // every lane has at most STEP_N_MAX entries; no steps otherwise
};

// Chain schedule of one strictly triangular factor (see trsv_chain): the
// rows of each slab are cut into tasks of at most TRSV_ROWS consecutive rows
// (in processing order: ascending for L, descending for U); consecutive tasks
// whose first row depends on the previous task's last row form a strand,
// which one warp solves task after task with that dependency held in
// registers.  Strands are dealt to the warps of the slab's CTA in a
// topological order of the strand graph, so every wait ends.
template <typename TV>
struct ChainHost {
  EllHost<TV> ell;            // per-slab ELL; an entry resolved in registers carries col = -2 - d,
                              // d = distance back in the warp's processing order (1..TRSV_ROWS)
  std::vector<int32_t> wptr;  // per slab: NWARP + 1 offsets into task (warp w: [wptr[w], wptr[w+1]))
  std::vector<int32_t> task;  // per task: first row processed, rows | (sequential ? 8 : 0)
  int64_t nstrands = 0;
};

template <typename TV>
struct SellSet {
  SellHost<TV> A;
  SellHost<double> A64;
  EllHost<TV> L, U;      // strictly lower / upper parts, slab-major order
  std::vector<TV> diag;  // npad: reciprocal pivots 1 / L_ii, 1 on padding rows
};

// 0 on success; 2 = malformed CSR, 3 = non-positive diagonal (msg says why).
int validate_csr(int64_t n, int64_t nnz, const int64_t *rp, const int32_t *ci, const double *va, std::string &msg);

// IC(lfil, tau) of A plus the levels of L and L^T.  0 on success, -2 on a
// non-positive pivot (column in *bad_col).
int ic_factor_host(int64_t n, const int64_t *rp, const int32_t *ci, const double *va, int lfil, double tau,
                   Factor &F, int64_t *bad_col);
// The factor from L by columns (column k: entries cs[k]..cs[k+1]-1 of
// rows/vals, diagonal first, rows ascending): L by rows and the levels.
void factor_from_columns(int64_t n, std::vector<int64_t> cs, std::vector<int32_t> rows, std::vector<double> vals,
                         Factor &F);

// Greedy multicolour ordering (nle_multicolor_order in nle.h): perm[new] =
// old, rows by colour then by row.  Returns the number of colours.
int32_t multicolor_order(int64_t n, const int64_t *rp, const int32_t *ci, int distance, std::vector<int32_t> &perm);
// B = P A P^T (perm[new] = old) in CSR with ascending columns in every row.
void permute_csr(int64_t n, const int64_t *rp, const int32_t *ci, const double *va, const std::vector<int32_t> &perm,
                 std::vector<int64_t> &brp, std::vector<int32_t> &bci, std::vector<double> &bva);
// perm[new] = old: rows cut into slabs of bsize consecutive values of
// locality[row] (the row itself when locality is NULL; locality must be a
// permutation of 0..n-1); inside a slab, by level of L, then by locality.
// P L P^T stays lower triangular.
void slab_level_order(const Factor &F, int64_t bsize, const int32_t *locality, std::vector<int32_t> &perm,
                      std::vector<int32_t> &iperm);

void permute(int64_t n, const int64_t *rp, const int32_t *ci, const double *va, const Factor &F,
             const std::vector<int32_t> &perm, const std::vector<int32_t> &iperm, int64_t npad, Permuted &P);

// level_rounds: split every group of R rows (the rows a warp of the level
// schedule takes at a time, 4 or 2) into one round per level (needed when
// dependencies can point to later slabs; see trsv_block).
template <typename TV>
void build_sell(const Permuted &P, int H, int64_t bsize, bool level_rounds, int R, SellSet<TV> &S,
                bool with_ell = true, bool with_a = true);

// Run a and b, set-up work on n rows, a on a thread of its own where that pays
// and one can be had.  An exception of either leaves only after both have ended.
// Below THREAD_ROWS a thread costs more than it saves: set-up of 100 rows, fixed
// schedule, 0.72 ms without threads, 0.88 with, of 1,110 rows 2.29 and 2.37; at 4,200 rows the
// set-up with threads takes what it took before there were any (4.8 ms).
constexpr int64_t THREAD_ROWS = 4096;
template <typename FA, typename FB>
void both(int64_t n, FA a, FB b) {
  std::future<void> f;
  if (n < THREAD_ROWS) {
    a();
  } else {
    try {
      f = std::async(std::launch::async, [&a] { a(); });
    } catch (const std::system_error &) {
      a();
    }
  }
  b();
  if (f.valid()) f.get();
}

// Steps of the strictly lower (lower = true) or upper factor for solve slabs of
// `rows` rows, with lpr (1, 2, 4 or 8) lanes per row and nwarps warps.
// plan_steps cuts the steps and collects the halo of every solve slab, unless
// a row is too long (out.fits = false, no steps); build_steps then fills in operands and coefficients for a window of own
// results from element 0, the zero at element `rows` and the halo behind it.
template <typename TV>
void plan_steps(const Permuted &P, int64_t rows, bool lower, int lpr, int nwarps, StepsHost<TV> &out);
template <typename TV>
void build_steps(const Permuted &P, int64_t rows, bool lower, int lpr, StepsHost<TV> &out);

// Forecast of one solve in us, step form and polled form, for a plan with one
// slab per solve slab: the steps of a plan, level by level, with the costs of
// FormCost.  A level of a slab begins when the level before it is done and the values
// it needs of other slabs are there.
struct FormCost {
  double level, next, hop, halo, quad, nquad;     // step form: first step of a level, each further one, a value on its
                                                  // way to another slab, each halo value copied, each quad past the
                                                  // registers in the first step and in each further one
  double plevel, pgroup, phop, ppass, poverflow;  // polled form: a level, each further group of rows, a value on its
                                                  // way to another slab, a further pass of the warps over the level,
                                                  // an overflow step
};
struct Forecast {
  double steps, polled;
};
template <typename TV>
Forecast forecast(const Permuted &P, int64_t rows, bool lower, int lpr, int nwarps, int twarps,
                  const StepsHost<TV> &plan);

// Chain schedule of the strictly lower (lower = true: P.Lrp/Lcol/Lval, levels
// P.lev) or upper (P.Urp/Ucol/Uval, levels P.levU) factor for nwarps warps
// per slab.  Needs the identity relabelling (slabs are ranges of the
// factored matrix's own row order).
template <typename TV>
void build_chain(const Permuted &P, int64_t bsize, bool lower, int nwarps, ChainHost<TV> &out);

}  // namespace nle
