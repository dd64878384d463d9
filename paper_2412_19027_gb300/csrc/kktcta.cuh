// Small problems: the whole refined KKT solve, and the numeric factorization, by one
// CTA per problem of the cohort.
//
// The general path launches one or two kernels per elimination level and sweep and
// re-tests the refinement in a graph WHILE node; an MPC problem of order 900 has 40
// levels of fronts of about 24 rows, so a KKT solve was ~200 launches of 2 us kernels
// that use a fraction of one SM.  A problem whose fronts are all small and whose work
// vectors fit one SM's shared memory is instead taken through its levels by one CTA,
// a warp per front, with block barriers in the place of launches.  Every sum is formed
// in the order of the general kernels, so a problem's iterates are the same on either
// path, and the choice may depend on the cohort.  The two right-hand sides of an
// iteration that do not wait for each other (the constant and the affine one) take a
// CTA each.
//
// What bounds it now: one SM's FP64 pipe and the chain of pivots (a shuffle and an FMA,
// ~145 clocks, each), 640 of them one after the other in that problem.  MPC, T = 20, 8
// states, 3 inputs: a refined solve 1.0 -> 0.22 ms (two at once), a factorization 0.66 ->
// 0.40, the whole solve 22.0 -> 10.1 ms; 64 uneven ones 124 -> 47 ms.  With rows of ~100
// entries (one dense QP, n = 50) the residual's FP64 work fills the SM (6.1 ms; by launches
// 5.7), with thousands of fronts on a level their sweeps do: CtaCost has the line.
#pragma once

#include <vector>

#include "device.cuh"
#include "scal.cuh"
#include "symbolic.h"

namespace clr {

// Longest source list that is summed entry by entry in list order; beyond, by the trees
// of k_pull_long.  A line of compatibility (see kThinCount): sums up to here keep the order
// they had.  From ~500 sources on (portfolio, entropy) the serial chain is what the level
// waits for.
constexpr int64_t kPullSerial = 512;
// The solves' lists of more than this many sources are read by a warp (in order up to
// kPullSerial), the longer ones by a CTA; the factor's lists, as many as a front's
// entries, stay a thread each up to kPullSerial and go to a warp beyond.
constexpr int64_t kSvThread = 32, kFaWarp = 8192;

// One front, in (problem, level) order.  Slots, positions and rows are relative to the
// problem's first.
struct alignas(16) CtaFront {
  int64_t goff;          // front (f x f, column-major) in the frontal pool
  int32_t c, f;          // pivots, rows
  int32_t woff;          // first solve slot
  int32_t pos;           // elimination position of the first pivot
  int32_t rows;          // update rows' positions: rows_loc[rows .. rows + f - c)
  int32_t pull0, npull;  // its solve pull targets
  int32_t nfa;           // its extend-add pull targets: [fa0, fa0 + nfa)
  int64_t fa0;
  int64_t pad;
};

// One solve pull target: its slot and sources (slots relative to the problem's first);
// sources past the fourth at pl_src[more ..].
struct alignas(16) CtaPull {
  uint16_t tg, n, s[4];
  int32_t more;
};

struct CtaProblem {
  int32_t lev0, nlev;  // its levels: fronts lev_ptr[lev0 + l] .. lev_ptr[lev0 + l + 1]
  int32_t pos0, N;     // its elimination positions
  int64_t w0;          // first solve slot (cohort)
  int32_t wtot;
  int32_t wide;        // its front of more than kCtaStage column entries (at most one), or -1
};

// Device arrays of the plan (n == 0: the cohort does not qualify).
struct CtaPlan {
  int64_t n = 0;  // problems
  const CtaProblem* prob = nullptr;
  const CtaFront* front = nullptr;
  const int32_t* lev_ptr = nullptr;  // per level: first front
  const int32_t* rows_loc = nullptr;
  const CtaPull* pull = nullptr;    // solve pulls, front by front
  const int32_t* pl_src = nullptr;
  const int32_t* perm = nullptr;    // KKT index of each elimination position
  const int32_t* slot = nullptr;    // solve slot of each elimination position (local)
  const int32_t* w_init = nullptr;  // KKT index of each solve slot's right-hand side, or -1
  int32_t max_slots = 0;            // largest wtot + N
  int32_t max_front = 0, max_cols = 0, max_wide = 0, max_levels = 0;  // largest f, staged and wide c f, levels
  bool factor = false;                                  // the factorization qualifies too
};
constexpr int kCtaRows = 96;               // largest front of the solves
constexpr int kCtaWarpRows = 32;           // largest front of the factorization: a row per lane
constexpr int kCtaStage = 640;             // largest c f copied ahead into a warp's buffers
constexpr int kCtaThreads = 512;
constexpr int kCtaSweepWarps = 8;          // warps that sweep fronts (two column buffers each)
constexpr int64_t kCtaSmem = 220 * 1024;   // shared memory of a CTA
constexpr int64_t kCtaWork = 1 << 18;      // factor entries, and KKT entries, of a problem one CTA takes

// When a CTA per problem is faster than a launch per level (the results are the same bits, so the choice
// may depend on the cohort).  A problem's fronts are one SM's work here and the whole GPU's there: a
// separable QP of 4000 variables, one level of 4000 fronts of 3 rows, took 32.4 ms on one CTA and 3.6 ms by
// launches; a dense QP of n = 72, one front of 93 rows swept by one warp, 11.1 and 8.9 ms; MPC, T = 20,
// 11.6 and 21.4 ms; 64 dense QPs of n = 50 in one cohort, 9.7 and 12.4 ms.  The times are estimated
// at setup, in microseconds, by constants fitted to per-iteration times on a GB300 (FP64; 57 cohorts:
// separable, box, total-variation chains and grids, dense QPs, MPC, 1 .. 200 problems).  Over these the
// choice costs 4 % of the solves' time at worst (dense QP, n = 40, where both are even).
struct CtaCost {
  std::vector<double> sweep;   // per problem: one right-hand side's two sweeps by its CTA, the residual but for its entries
  double levels = 0;           // the same by launches, whole cohort
  double factor = 0, factor_levels = 0;
};
// the refined solves of an iteration (two launches for three right-hand sides); entries: KKT entries of each problem
bool cta_solve_pays(const CtaCost& c, const std::vector<int64_t>& entries);

// Host: the plan of a cohort whose fronts are all of at most kCtaRows rows, or n = 0.
int cta_plan_build(DeviceArena& ar, const Symbolic& sy, const NumericMaps& mp, int small_max,
                   const std::vector<int32_t>* pos_pid, const int32_t* d_w_init, CtaPlan& out, CtaCost& cost);

// One right-hand side of a launch: its solution and residual vectors (KKT order).
struct CtaRhs {
  const double* rhs;
  double *sol, *r;
};
// Refinement state of one solve (the fields of IterScal that the test works on).
struct IrState {
  int ir_skip, ir_cur, ir_total, ir_revert, ir_fail;
  double rhs_norm, ir_prev, ir_worst;
  unsigned long long rnorm_bits;
};

// Refinement constants (Sec. 3.6).
struct IrParams {
  double abstol, reltol, stop_ratio;
  int max_steps;
};
// The KKT matrix (full CSR) as the residual reads it.
struct KmvArgs {
  int64_t n;
  const int64_t* kptr;
  const int32_t *kcol, *kvi;
  const double *kval, *kfv;
  const int4* krow;  // the rows of each problem in turn (from its pos0), shortest class first: KKT row,
                     // first and past-the-last entry
  const int32_t* kcls;  // per problem kKrowClasses ends of the row classes in its list
};
// Row length classes of the residual: at most 1, 2, 4, 8, 16, 32 entries, more.
constexpr int kKrowClasses = 7;
inline int krow_class(int64_t len) {
  int c = 0;
  while (c < kKrowClasses - 1 && len > ((int64_t)1 << c)) ++c;
  return c;
}

template <typename T>
struct CtaOps {
  static int setup_attributes();
  // the extend-adds and partial factorizations of every level (fronts scattered and regularised before)
  static int factor(cudaStream_t st, const CtaPlan& cp, T* F, T* Dp, const int8_t* dsign, const int64_t* fa_tgt,
                    const int64_t* fa_ptr, const int64_t* fa_src, double eps, double delta, int* hits,
                    const int* skip);
  // the refined solves of one or two right-hand sides (b.rhs null: one), a CTA each
  static int kkt_solve(cudaStream_t st, const CtaPlan& cp, const KmvArgs& k, const T* F, const T* Dp, const CtaRhs& a,
                       const CtaRhs& b, IterScal* sc, const IrParams& ir, const int* skip);
};

}  // namespace clr
