// Row sums of the K product and the refinement test, shared by the per-kernel path
// (ipm.cu) and the one-CTA-per-problem path (kktcta.cu).
#pragma once

#include "device.cuh"
#include "scal.cuh"

namespace clr {

__device__ __forceinline__ unsigned long long dbits(double v) { return (unsigned long long)__double_as_longlong(v); }
__device__ __forceinline__ double bitsd(unsigned long long b) { return __longlong_as_double((long long)b); }

// Entry p of row i, column c.  kfv holds the constant values (P and A) in row order; the
// z-z block's, which change from iteration to iteration, are read through the value index.
__device__ __forceinline__ double kmv_value(int64_t i, int64_t p, int32_t c, int64_t n, const int32_t* __restrict__ kvi,
                                            const double* __restrict__ kval, const double* __restrict__ kfv) {
  return i >= n && c >= n ? kval[kvi[p]] : kfv[p];
}
// Sum of the lanes' partials, lanes outside `used` holding 0: the tree t += t + 16, ..., and for
// one partial what the tree gives, x + 0.
__device__ __forceinline__ double kmv_tree(double a, unsigned used) {
  if (used == 0) return 0.0;
  if ((used & (used - 1)) == 0) return __dadd_rn(__shfl_sync(0xffffffffu, a, __ffs(used) - 1), 0.0);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) a = __dadd_rn(a, __shfl_xor_sync(0xffffffffu, a, off));
  return a;
}
// Entries [s0, s1) of row i by a warp, entry p to lane (p - s0) mod 32.  An FP64 instruction
// takes 64 clocks of its pipe however few lanes are active, so sums that no lane adds to are left out
// (a row's columns are sorted: most steps have one kind).
__device__ __forceinline__ void kmv_warp(int64_t i, int64_t s0, int64_t s1, int64_t n, const int32_t* __restrict__ kcol,
                                         const int32_t* __restrict__ kvi, const double* __restrict__ kval,
                                         const double* __restrict__ kfv, const double* v, int lane, double& a, double& b,
                                         unsigned& ua, unsigned& ub) {
  a = b = 0.0;
  ua = ub = 0;
  for (int64_t base = s0; base < s1; base += 128) {
    double x[4], y[4];
    int32_t c[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t p = base + 32 * k + lane;
      c[k] = p < s1 ? kcol[p] : -1;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      x[k] = c[k] >= 0 ? kmv_value(i, base + 32 * k + lane, c[k], n, kvi, kval, kfv) : 0.0;
      y[k] = c[k] >= 0 ? v[c[k]] : 0.0;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const unsigned ma = __ballot_sync(0xffffffffu, c[k] >= 0 && c[k] < n);
      const unsigned mb = __ballot_sync(0xffffffffu, c[k] >= n);
      if ((ma | mb) == 0) break;
      const double t = __dmul_rn(x[k], y[k]);
      if (ma) a = c[k] >= 0 && c[k] < n ? __dadd_rn(a, t) : a;
      if (mb) b = c[k] >= n ? __dadd_rn(b, t) : b;
      ua |= ma;
      ub |= mb;
    }
  }
}

// Sums of row i (entries p0 .. p1) by G lanes: a over the columns < n, b over the
// others, valid in lane 0 of the group.  32 partial sums, entry e of the row going to
// partial e mod 32, then the pairwise tree t += t + 16, t += t + 8, ..., whatever G is.
template <int G>
__device__ __forceinline__ void kmv_row(int64_t i, int64_t p0, int64_t p1, int64_t n, const int32_t* __restrict__ kcol,
                                        const int32_t* __restrict__ kvi, const double* __restrict__ kval,
                                        const double* __restrict__ kfv, const double* v, int lane, unsigned gmask,
                                        double& ra, double& rb) {
  if constexpr (G == 32) {
    unsigned ua, ub;
    double x, y;
    kmv_warp(i, p0, p1, n, kcol, kvi, kval, kfv, v, lane, x, y, ua, ub);
    ra = kmv_tree(x, ua);
    rb = kmv_tree(y, ub);
    return;
  }
  constexpr int NU = 32 / G;  // partial sums per lane: t = lane + G u
  double a[NU], b[NU];
#pragma unroll
  for (int u = 0; u < NU; ++u) a[u] = b[u] = 0.0;
  // four 32-entry steps per pass: all loads of the pass issued before the adds,
  // which keep the order of the plain one-step loop (partial t sums entries
  // p = p0 + t (mod 32) in increasing p)
  for (int64_t base = p0; base < p1; base += 128) {
    double tv[4][NU];
    bool tx[4][NU];
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int u = 0; u < NU; ++u) {
        const int64_t p = base + 32 * k + lane + G * u;
        tv[k][u] = 0.0;
        tx[k][u] = true;
        if (p < p1) {
          const int32_t c = kcol[p];
          tv[k][u] = kmv_value(i, p, c, n, kvi, kval, kfv) * v[c];
          tx[k][u] = c < n;
        }
      }
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int u = 0; u < NU; ++u) {
        if (base + 32 * k + lane + G * u >= p1) continue;
        if (tx[k][u]) a[u] += tv[k][u];
        else b[u] += tv[k][u];
      }
  }
#pragma unroll
  for (int off = 16; off >= G; off >>= 1)
#pragma unroll
    for (int u = 0; u < off / G; ++u) {
      a[u] += a[u + off / G];
      b[u] += b[u + off / G];
    }
#pragma unroll
  for (int off = (G == 32 ? 16 : G / 2); off > 0; off >>= 1) {
    a[0] += __shfl_xor_sync(gmask, a[0], off, G);
    b[0] += __shfl_xor_sync(gmask, b[0], off, G);
  }
  ra = a[0];
  rb = b[0];
}

// The same two sums by one thread for a row of at most M entries (M a power of two up to
// 32): entry e is partial e, and the partials that are not there would only add zeros.
// An FP64 warp instruction takes 64 clocks of its pipe whatever its active lanes, so for
// one SM's worth of short rows a thread per row needs a fraction of the G-lane version's.
template <int M>
__device__ __forceinline__ void kmv_row_thread(int64_t i, int64_t p0, int64_t p1, int64_t n,
                                               const int32_t* __restrict__ kcol, const int32_t* __restrict__ kvi,
                                               const double* __restrict__ kval, const double* __restrict__ kfv,
                                               const double* v, double& ra, double& rb) {
  double a[M], b[M];
#pragma unroll
  for (int e = 0; e < M; ++e) {
    a[e] = b[e] = 0.0;
    const int64_t p = p0 + e;
    if (p < p1) {
      const int32_t c = kcol[p];
      const double t = kmv_value(i, p, c, n, kvi, kval, kfv) * v[c];
      if (c < n) a[e] = t;
      else b[e] = t;
    }
  }
#pragma unroll
  for (int off = M / 2; off > 0; off >>= 1)
#pragma unroll
    for (int e = 0; e < off; ++e) {
      a[e] = __dadd_rn(a[e], a[e + off]);
      b[e] = __dadd_rn(b[e], b[e + off]);
    }
  ra = a[0];
  rb = b[0];
}

// Refinement test of one problem (Sec. 3.6): stop at the tolerance, or after
// max_steps steps, or, when stop_ratio > 0 and ||r||_inf is already below the
// acceptance bar fail_tol = 1e-4 max(1, ||rhs||_inf), as soon as a step has
// reduced ||r||_inf by less than stop_ratio (the last correction is kept).  A
// step that made ||r||_inf larger is undone (k_ir_revert) and ends the
// refinement: the regularised factor is not a contraction for K there.
// A refinement that ends above fail_tol marks the iteration (ir_fail = 1; 2 if
// the residual is not finite): with a low-precision factor it is then redone in
// FP64; in FP64 a non-finite solve stops the solve at the current iterate.
// (S: IterScal, or one solve's own copy of its refinement fields.)
template <typename S>
__device__ __forceinline__ bool ir_step_due(S& q, double abstol, double reltol, double stop_ratio, int max_steps) {
  const double r = bitsd(q.rnorm_bits);
  q.rnorm_bits = 0ull;
  q.ir_revert = 0;
  if (q.ir_skip) return false;
  const double fail_tol = 1e-4 * fmax(1.0, q.rhs_norm);
  const double tol = abstol + reltol * q.rhs_norm;
  if (r > q.ir_prev) {
    q.ir_revert = 1;
    q.ir_skip = 1;
    if (!(q.ir_prev <= fail_tol)) q.ir_fail = max(q.ir_fail, isfinite(q.ir_prev) ? 1 : 2);
    if (q.ir_prev > tol) q.ir_worst = fmax(q.ir_worst, q.ir_prev);
    return false;
  }
  const bool stalled = stop_ratio > 0 && r <= fail_tol && !(r * stop_ratio < q.ir_prev);
  q.ir_prev = r;
  if (!(r > tol) || stalled || q.ir_cur >= max_steps) {  // NaN also stops
    q.ir_skip = 1;
    if (!(r <= fail_tol)) q.ir_fail = max(q.ir_fail, isfinite(r) ? 1 : 2);  // 2: a non-finite solve
    if (r > tol) q.ir_worst = fmax(q.ir_worst, r);
    return false;
  }
  q.ir_cur += 1;
  q.ir_total += 1;
  return true;
}

}  // namespace clr
