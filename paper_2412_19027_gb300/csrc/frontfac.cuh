// Partial LDL^T of one small front by a group of warps, in registers.
#pragma once

#include "device.cuh"

namespace clr {

template <typename T>
__device__ __forceinline__ T regularise(T d, int sgn, T eps, T delta, bool* hit) {
  if ((T)sgn * d <= eps) {
    *hit = true;
    return (T)sgn * delta;
  }
  *hit = false;
  return d;
}
// s - (a b) inv, the elimination step of one front entry
__device__ __forceinline__ double elim(double s, double a, double b, double inv) { return fma(-(a * b), inv, s); }
__device__ __forceinline__ float elim(float s, float a, float b, float inv) { return fmaf(-(a * b), inv, s); }
__device__ __forceinline__ double rcp_exact(double d) { return __drcp_rn(d); }  // = 1 / d, rounded to nearest
__device__ __forceinline__ float rcp_exact(float d) { return __frcp_rn(d); }
__device__ __forceinline__ double flip(double x, bool neg) {  // neg ? -x : x without an FP64 instruction
  return __hiloint2double(__double2hiint(x) ^ (neg ? (int)0x80000000 : 0), __double2loint(x));
}
__device__ __forceinline__ float flip(float x, bool neg) {
  return __int_as_float(__float_as_int(x) ^ (neg ? (int)0x80000000 : 0));
}

// Shared memory of a front of f rows, in elements: the front, its pivots, their
// reciprocals and expected signs.
__host__ __device__ constexpr int front_words(int f) { return f * f + 3 * f; }

// Partial LDL^T (c pivots) of the front of f rows held at S (f x f, column-major; front_words(f)
// elements) by GW warps, results to G and Dp.  Per pivot k: d = S_kk, replaced by sign delta
// when sign d <= eps; S_ij -= (S_ik S_jk) / d for i >= j > k with the exact reciprocal; then
// column k is scaled.
//
// Bound by the pivots' chain (barrier, reciprocal 354 clocks) and by FP64 warp instructions
// (64 clocks each): the lower entries sit in registers, NS a lane in column-major order, so
// that an instruction has 32 useful lanes and a slot whose columns are done is skipped, only
// the next pivot column goes through shared memory, one barrier per pivot, and the columns are
// scaled once at the end.  (A full square of entries per pivot, a division per thread and three
// barriers before: 16 us for a level of 24-row fronts of 16 pivots, 10 now; the factorization
// of a dense QP with a root of 65 pivots 136 -> 105 us.)
template <typename T, int NS, int GW>
__device__ __forceinline__ void factor_regs(T* S, T* G, T* Dp, const int8_t* dsign, int c, int f, T eps, T delta,
                                            int* hits, int bar) {
  constexpr int NL = 32 * GW;
  const int t = threadIdx.x & (NL - 1), E = f * (f + 1) / 2;
  auto sync = [&]() {
    if constexpr (GW == 1) __syncwarp();
    else asm volatile("barrier.sync %0, %1;" ::"r"(bar), "n"(NL) : "memory");
  };
  T* sd = S + f * f;
  T* si = sd + f;
  int8_t* sg = reinterpret_cast<int8_t*>(si + f);
  for (int k = t; k < c; k += NL) sg[k] = dsign[k];
  T v[NS];
  int rc[NS];  // column << 16 | row (-1: no entry)
  int row = t, col = 0;
  sync();  // S is complete
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    while (row >= f && col < f) {  // past the end of column col: on from the next one's diagonal
      row += col + 1 - f;
      ++col;
    }
    const bool in = NL * s + t < E;
    rc[s] = in ? (col << 16 | row) : -1;
    v[s] = in ? S[row + col * f] : (T)0;
    row += NL;
  }
  for (int k = 0; k < c; ++k) {
    sync();
    T d = S[k + k * f];
    const bool ng = sg[k] < 0;
    const bool hit = flip(d, ng) <= eps;  // sign * d <= eps
    if (hit) d = flip(delta, ng);
    const T inv = rcp_exact(d);
    if (t == 0) {
      if (hit) atomicAdd(hits, 1);
      sd[k] = d;
      si[k] = inv;
    }
    const int st = (k + 1) * f - (k + 1) * k / 2;  // first entry of column k + 1
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      if (NL * s + NL - 1 < st || NL * s >= E) continue;
      const int q = rc[s] >> 16, r = rc[s] & 0xffff;
      if (q > k) {
        v[s] = elim(v[s], S[r + k * f], S[q + k * f], inv);
        if (q == k + 1) S[r + q * f] = v[s];
      }
    }
  }
  sync();
  // the columns of L (their unscaled entries are in S), the pivots, the update block
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    if (rc[s] < 0) continue;
    const int q = rc[s] >> 16, r = rc[s] & 0xffff;
    G[r + q * f] = q >= c ? v[s] : (r == q ? sd[q] : S[r + q * f] * si[q]);
  }
  for (int k = t; k < c; k += NL) Dp[k] = sd[k];
  sync();
}
template <typename T, int GW>
__device__ __forceinline__ void factor_front32(T* S, T* G, T* Dp, const int8_t* dsign, int c, int f, T eps, T delta,
                                               int* hits, int bar) {
  constexpr int A = (136 + 32 * GW - 1) / (32 * GW), B = (300 + 32 * GW - 1) / (32 * GW),
                C = (528 + 32 * GW - 1) / (32 * GW);
  if (f <= 16) factor_regs<T, A, GW>(S, G, Dp, dsign, c, f, eps, delta, hits, bar);
  else if (f <= 24) factor_regs<T, B, GW>(S, G, Dp, dsign, c, f, eps, delta, hits, bar);
  else factor_regs<T, C, GW>(S, G, Dp, dsign, c, f, eps, delta, hits, bar);
}

}  // namespace clr
