// Numeric supernodal (multifrontal) LDL^T of the quasi-definite KKT matrix
// and its level-scheduled triangular solves (Sec. 3.6 of the paper, Alg. 1
// steps 5, 6 and 9).  T is the factor precision (double or float).
#pragma once

#include <vector>

#include "bigfront.cuh"
#include "thinsyrk.cuh"
#include "device.cuh"
#include "internal.h"
#include "kktcta.cuh"
#include "scal.cuh"
#include "symbolic.h"

namespace clr {

// Device arrays of the symbolic structure and the index maps (shared by the
// FP64 and FP32 factors).
struct LdlStructure {
  int64_t N = 0, nsn = 0, nlev = 0, pool = 0, wtot = 0, nk = 0;
  int64_t *sn_ptr = nullptr, *row_ptr = nullptr, *front_off = nullptr, *upd_off = nullptr, *lev_sn = nullptr;
  int32_t* rows_kkt = nullptr;
  int32_t* w_init = nullptr;   // solve slot -> KKT index of the right-hand side, or -1
  int8_t* dsign = nullptr;     // expected pivot sign by position
  int32_t* pos_pid = nullptr;  // problem of each elimination position (cohorts)
  int64_t *kdest = nullptr, *diag_pos = nullptr;
  int64_t *fa_tgt = nullptr, *fa_ptr = nullptr, *fa_src = nullptr;
  int64_t *sv_tgt = nullptr, *sv_ptr = nullptr, *sv_src = nullptr;
  // host copies used to configure launches
  std::vector<int64_t> h_lev_ptr, h_lev_sn, h_fa_lev_ptr, h_sv_lev_ptr;
  std::vector<int64_t> h_sn_ptr, h_row_ptr, h_front_off;
  std::vector<int> lev_small_maxf;               // largest small front of each level
  // fronts by kernel, per level (device lists): small ones (one CTA each in shared
  // memory), thin ones without and with children (ldl_thin_front), and both kinds
  // together (the solves' one CTA per front)
  struct List {
    const int64_t* id = nullptr;
    int64_t n = 0;
    int64_t first = 0;  // lev_cta: index of its first entry in cta_pull
  };
  std::vector<List> lev_small, lev_thin_leaf, lev_thin, lev_cta;
  std::vector<List> lev_thin_syrk;               // thin leaves whose update matrices are a product (thinsyrk.cu)
  ThinSyrk syrk;
  bool f64 = false;                              // the factor is FP64 (set before ldl_structure_upload)
  bool f64_later = false;                        // an FP64 factor may take over (likewise)
  std::vector<int64_t> lev_thin_smem;            // largest f c of a level's thin fronts
  // pull targets with long source lists (indices into fa_tgt, sv_tgt): a warp each (the solves'
  // in list order), a CTA each
  std::vector<List> fa_warp, fa_cta, sv_warp, sv_cta;
  std::vector<std::vector<int64_t>> lev_big;     // big fronts of each level
  BigFrontDev bfd;                               // big-front arrays (device)
  std::vector<BigLevelPlan> bplans;              // per level
  std::vector<SweepLevel> sweeps;                // per level: the solve sweeps over its big fronts
  std::vector<int8_t> lev_fused;                 // per level: the forward kernels gather the children themselves
  int32_t* pull_ptr = nullptr;                   // big fronts of fused levels: pull target of each row, or -1
  int64_t* cta_pull = nullptr;                   // per lev_cta entry: its pull targets' range (two words)
  // extend-add by relative indices: per level, the rounds' work lists (children
  // and prefix sums of their 32 x 32 tile counts)
  int32_t* rel = nullptr;
  int64_t* rel_off = nullptr;
  int64_t* sn_parent = nullptr;
  std::vector<std::vector<WorkList>> push_rounds;
  // dataflow factorization of the big fronts: task table (device), per level
  // its task range and the offset of its task counter in the state words;
  // per big-front id the offset of its version words
  FlowTask* flow_task = nullptr;
  int64_t* flow_soff = nullptr;
  std::vector<int64_t> flow_t0, flow_nt, flow_head;
  std::vector<int8_t> flow_one;  // per level: launch one CTA per SM (else two)
  std::vector<int8_t> flow_tc;   // per level: FP32 factors use the tensor-core launch
  // the FP64 factor's task table (the fused chain task split, bigfront.cuh), per level
  FlowTask* flow_task64 = nullptr;
  // the FP64 fronts whose products run on the tensor cores (bigflow64.cu): their table, per level
  // its range and counter; flow_emu: allowed (set before ldl_structure_upload)
  bool flow_emu = true;
  FlowTask* flow_task64e = nullptr;
  struct Flow64Launch {
    int64_t t0, nt, head;
  };
  std::vector<std::vector<Flow64Launch>> flow_64e;  // per level, one after the other (they share the packs' space)
  int64_t flow_head64e = 0;     // their counters: one word per front with digit products, from here on
  int64_t pk64_tiles = 0;       // digit packs of the largest launch
  int64_t pk64_front = 0;       // ... of the largest front
  bool pk64_no_room = false;    // the packs did not fit: FMA products
  std::vector<int64_t> h_bf_f, h_bf_c, h_bf_lev;  // big fronts: rows, pivots, level
  std::vector<int64_t> flow_t0_64, flow_nt_64;
  std::vector<int8_t> flow_one64;
  int64_t flow_words = 0;
  int64_t pk_tiles = 0;  // packed operand tiles of the largest level (tensor-core flow, FP32 factor)
  int small_max = 0;
  int64_t max_front = 0;
  CtaPlan cta;  // small problems: a CTA per problem (n = 0: not used)
  CtaCost cta_cost;
};

// A front of more rows than small_max with few pivots: the arrow columns of a dense
// row block (portfolio, Huber, entropy problems have thousands with 1 .. 5 pivots and
// hundreds of rows).  Its update matrix is a rank-c product that one CTA streams out
// (k_factor_thin); cut into 64 x 64 tile tasks of the dataflow launch, a task did
// 1/64 .. 1/16 of a tile's work for the same loads, stores and waits (portfolio
// n = 5000, FP32: 5000 fronts of ~250 rows 3.0 -> 0.20 ms), and the forward sweep
// gave each front f / 32 CTAs of 512 threads for one or two columns (100 -> 9 us).
// The lines: f^2 c / 2 FMAs on one SM are 0.3 ms in FP64 at 2^21, about what the tile
// tasks of one such front take end to end.  A problem with fewer than kThinCount of them
// keeps the tile tasks.  That line, like those of kPullSerial and kFlow64Rows, is one of
// compatibility and not where the times cross: with the three at 8 fronts, 48 sources and
// 96 rows a factorization with fronts of 151 rows and one pivot took 0.44 ms in the place
// of 0.69 for 32 of them and 0.55 for 1.02 with 500 (FP64; FP32 0.16 for 0.17 and 0.17 for
// 0.47), but dense QPs up to n ~ 250, which have such fronts too, would give other last
// digits of their multipliers (1e-9) than before.  The rule looks at one problem, so that
// its arithmetic does not depend on its cohort.
constexpr int64_t kThinPivots = 16, kThinWork = (int64_t)1 << 21, kThinCount = 512;
inline bool ldl_thin_front(int64_t f, int64_t c, int small_max) {
  return f > small_max && c <= kThinPivots && f * f * c <= kThinWork;
}

// Which kernels a structure's fronts take (clr_get_routes).
void ldl_routes(const LdlStructure& st, clr_routes* out);

// pos_pid: problem of each elimination position (null: one problem).
int ldl_structure_upload(DeviceArena& ar, const Symbolic& sy, const NumericMaps& mp, const std::vector<int8_t>& dsign,
                         int small_max, LdlStructure& st, const std::vector<int32_t>* pos_pid = nullptr);

template <typename T>
struct LdlFactor {
  const LdlStructure* s = nullptr;
  T* F = nullptr;   // frontal-matrix pool
  T* Dp = nullptr;  // pivots by elimination position
  T* w = nullptr;   // forward-solve slots
  T* xs = nullptr;  // solution in KKT order
  T* E = nullptr;     // augmented inverse blocks of the big fronts
  T* ybuf = nullptr;  // forward results of the big fronts
  T* Linv = nullptr;  // per big front, two 64 x 64 diagonal-block inverses
  int* dyn_hits = nullptr;
  int* tc_err = nullptr;  // set if a wait of the big-front kernels ran out (the factor is unusable)
  bool tc16 = false;      // big-front updates with BF16 products on the tensor cores (float only)
  bool flow = true;       // big fronts by the dataflow kernel (one launch per level); else per-panel launches
  int flow_tc = 1;        // FP32 dataflow, trailing and E updates on the tensor cores (TF32 hi/lo parts):
                          // 0 never, 1 on the levels whose simulated schedule is shorter that way, 2 always
  T *syrk_w = nullptr, *syrk_part = nullptr;  // panels and partial tiles of thinsyrk.cu
  unsigned char* pk64 = nullptr;  // FP64: digit packs of the largest launch (null: FMA products on every front)
  FlowTc tcs;             // its packed operand tiles and their tensor map (allocated when used)
  int* flow_state = nullptr;
  int flow_sms = 0, flow_occ = 0;  // SMs of the device, resident flow CTAs per SM
  int alloc(DeviceArena& ar, const LdlStructure& st);
  // The digit packs of an FP64 factor, after everything else that the owner allocates: without room for
  // a launch's packs the fronts go one at a time (the same results), without room for one front's with FMA
  // products.
  int alloc_packs(DeviceArena& ar, LdlStructure& st);
  // the FP32 dataflow factorization with tensor-core updates is in use
  bool use_flow_tc() const { return sizeof(T) == 4 && flow && flow_tc != 0 && !tc16 && s && s->pk_tiles > 0; }
  // Factor K: kval (FP64, lower triangle entries in kval order) scattered into
  // the fronts, +/- delta added on the diagonal (x rows +, z rows -), with
  // delta = sc[p].delta of the position's problem p.
  int factor(cudaStream_t st, const double* kval, const IterScal* sc, double dyn_eps, double dyn_delta,
             const int* skip) const;
  // xs = (L D L^T)^{-1} rhs (rhs FP64 in KKT order).
  int solve(cudaStream_t st, const double* rhs, const int* skip) const;
};

}  // namespace clr
