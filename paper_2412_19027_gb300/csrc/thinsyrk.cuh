// Many thin leaf fronts of one parent: extend-add as a product, solves by their columns (thinsyrk.cu).
#pragma once

#include <cstdint>
#include <vector>

#include "device.cuh"
#include "symbolic.h"

namespace clr {

struct ThinSyrkParent {
  int64_t goff, fP, ld;     // the parent's front in the pool, its rows; row length of its panel W
  int64_t K, col0, woff;    // columns of its thin leaves, the first one in the column arrays, W's offset
  int64_t tiles, splits, kc;
  int64_t wslot;            // the parent's work vector
  int64_t front0, nfront;   // its leaves in `front`
  int64_t vsplits, vc;      // columns per split of the solve's product
  int32_t many;             // a leaf has several pivots
};

struct ThinSyrk {
  std::vector<std::vector<ThinSyrkParent>> lev;  // by the parent's level
  std::vector<char> child;                       // host: fronts that keep no update matrix
  // per column: its rows below the pivots in the pool, how many, their places in the parent's
  // rows (first one in map), its pivot
  int64_t *src = nullptr, *map0 = nullptr;
  int32_t *cnt = nullptr, *dpos = nullptr, *map = nullptr;
  int64_t *slot = nullptr, *front = nullptr;     // per column: its pivot's place in the work vector; the leaves
  // parts of the pool that a factorization clears (offset, length <= kSegment): without the update
  // matrices that are not kept
  int64_t* seg = nullptr;
  int64_t nseg = 0;
  int64_t wtotal = 0, part = 0;                  // entries of all panels W; of the largest parent's partial tiles
};

// The extend-add or solve lists of a structure (NumericMaps' fa_*, sv_*), without what the products cover.
struct FaLists {
  std::vector<int64_t> lev_ptr, tgt, ptr, src;
};

// FMAs of the product per value that the lists would gather, at most, for FP64 and FP32 factors and for
// FP32 ones that may go on in FP64 with the same plan.  Factorization per iteration, product and lists, of
// the portfolio n = 5000 by the density of its factor matrix (FMAs per value):
//   FP32   0.50 and 2.01 ms at 8.5, 0.49 and 1.55 at 12, 0.48 and 1.18 at 16, 0.51 and 0.88 at 23
//   FP64   4.69 and 11.8 ms at 2.1, 4.62 and 4.41 at 8.5, 4.60 and 3.54 at 12, 4.59 and 2.81 at 16, 4.58 and 2.10 at 23
// An FP32 iteration gains by the product what an FP64 one loses at about 12.  The FP64 line is on the safe
// side: between 2 and 7 the product would be faster.
constexpr int64_t kSyrkRatio64 = 2, kSyrkRatio32 = 64, kSyrkRatioBoth = 12;

// leaf: thin leaf fronts (ldl_thin_front, the path taken).  Chooses the parents, fills out and, if
// any was chosen, fa and sv.
int thin_syrk_plan(DeviceArena& ar, const Symbolic& sy, const NumericMaps& mp, const std::vector<char>& leaf, int64_t ratio,
                   int64_t min_children, ThinSyrk& out, FaLists& fa, FaLists& sv);

template <typename T>
struct ThinSyrkOps {
  static void clear_pool(cudaStream_t st, const ThinSyrk& ts, T* F);
  // F_P -= sum over the leaves' columns of l d l^T, for the parents of level l
  static void add_level(cudaStream_t st, const ThinSyrk& ts, int64_t l, T* F, const T* Dp, T* W, T* part,
                        const int* skip);
  // the leaves' forward sweep for the parents of level l: w_P -= sum over their columns of l y
  static void fwd_level(cudaStream_t st, const ThinSyrk& ts, int64_t l, const T* F, const T* W, T* part, T* w,
                        const int64_t* sn_ptr, const int64_t* row_ptr, const int64_t* front_off,
                        const int64_t* upd_off, const int* skip);
  // and their backward sweep, after the parents'
  static void bwd_level(cudaStream_t st, const ThinSyrk& ts, int64_t l, const T* F, const T* Dp, const T* w, T* xs,
                        const int64_t* sn_ptr, const int64_t* row_ptr, const int64_t* front_off,
                        const int64_t* upd_off, const int32_t* rows_kkt, const int* skip);
};
}  // namespace clr
