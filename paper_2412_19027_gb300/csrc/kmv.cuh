// Row sums of the K product and the refinement test, shared by the per-kernel path
// (ipm.cu) and the one-CTA-per-problem path (kktcta.cu).
#pragma once

#include "device.cuh"
#include "scal.cuh"

namespace clr {

__device__ __forceinline__ unsigned long long dbits(double v) { return (unsigned long long)__double_as_longlong(v); }
__device__ __forceinline__ double bitsd(unsigned long long b) { return __longlong_as_double((long long)b); }

// Sums of row i (entries p0 .. p1) by G lanes: a over the columns < n, b over the
// others, valid in lane 0 of the group.  32 partial sums, entry e of the row going to
// partial e mod 32, then the pairwise tree t += t + 16, t += t + 8, ..., whatever G is.
template <int G>
__device__ __forceinline__ void kmv_row(int64_t i, int64_t p0, int64_t p1, int64_t n, const int32_t* __restrict__ kcol,
                                        const int32_t* __restrict__ kvi, const double* __restrict__ kval,
                                        const double* __restrict__ kfv, const double* v, int lane, unsigned gmask,
                                        double& ra, double& rb) {
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
          tv[k][u] = (i < n ? kfv[p] : kval[kvi[p]]) * v[c];
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
      const double t = (i < n ? kfv[p] : kval[kvi[p]]) * v[c];
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
