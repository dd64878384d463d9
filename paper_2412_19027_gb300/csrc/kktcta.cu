// One CTA per small problem: numeric factorization and refined KKT solve (kktcta.cuh).
//
// Bound by latency: a level is a warp's chain of dependent L2 and shared accesses plus
// the pivots of its fronts (FP64 instructions at 64 clocks), then a barrier.
#include <algorithm>
#include <type_traits>

#include "frontfac.cuh"
#include "internal.h"
#include "kktcta.cuh"
#include "kmv.cuh"

namespace clr {

namespace {

// cp.async of n words of T from global to shared memory by a warp (8- or 4-byte copies: a
// front starts at any entry of the pool).
template <typename T>
__device__ __forceinline__ void warp_copy_async(T* dst, const T* src, int n) {
  const int lane = threadIdx.x & 31;
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  for (int q = lane; q < n; q += 32)
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d + (uint32_t)(q * sizeof(T))), "l"(src + q),
                 "n"(sizeof(T))
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_wait1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// The fronts a warp sweeps, level by level (up or down), its share of each level.
struct FrontSeq {
  const int32_t* lp;
  int nlev, step, wid, l, j;
  __device__ FrontSeq(const int32_t* lp_, int nlev_, int step_, int wid_)
      : lp(lp_), nlev(nlev_), step(step_), wid(wid_), l(step_ > 0 ? 0 : nlev_ - 1), j(0) {
    j = lp[l] + wid;
    settle();
  }
  __device__ bool done() const { return l < 0 || l >= nlev; }
  __device__ void settle() {
    while (!done() && j >= lp[l + 1]) {
      l += step;
      if (!done()) j = lp[l] + wid;
    }
  }
  __device__ void next() {
    if (done()) return;
    j += kCtaSweepWarps;
    settle();
  }
};

// Forward sweep of one front by a warp, a row per lane, its columns at Bf (f x c): the
// gather of k_pull and k_pull_warp, then the sums of k_fwd_front.  The triangle and the
// rows below it run through one FMA: lanes < c take L x_j off their entry, the others
// add it to a sum that is taken off at the end.  Two pivots a step: every lane forms the
// second one's value itself (one FMA) instead of waiting for another shuffle.
template <typename T>
__device__ __forceinline__ void fwd_front(const CtaPlan& cp, const CtaFront& m, const CtaPull& pl, const T* Bf, T* w) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, c = m.c, f = m.f;
  if (pl.n > 0) {
    T acc = w[pl.tg];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (u < pl.n) acc += w[pl.s[u]];
    for (int q = 4; q < pl.n; ++q) acc += w[cp.pl_src[pl.more + q - 4]];
    w[pl.tg] = acc;
  }
  __syncwarp();
  T* wj = w + m.woff;
  const bool in = lane < f, piv = lane < c;
  const T x0 = in ? wj[lane] : (T)0;
  T acc = piv ? x0 : (T)0;
  for (int j0 = 0; j0 < c; j0 += 8) {
    T v[8], d[4];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int j = j0 + u;
      v[u] = flip((j < c && in && lane > j) ? Bf[lane + j * f] : (T)0, piv);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) d[u] = j0 + 2 * u + 1 < c ? Bf[(j0 + 2 * u + 1) + (j0 + 2 * u) * f] : (T)0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = j0 + 2 * u;
      if (j >= c) break;
      const T xa = __shfl_sync(FULL, acc, j), xb0 = __shfl_sync(FULL, acc, j + 1 & 31);
      acc = v[2 * u] * xa + acc;
      if (j + 1 < c) {
        const T xb = xb0 - d[u] * xa;  // lane j + 1's own update by pivot j
        acc = v[2 * u + 1] * xb + acc;
      }
    }
  }
  if (in) wj[lane] = piv ? acc : x0 - acc;
}

// Backward sweep of one front by a warp after the division by D, the sums of k_bwd_front:
// lane r holds row c + r below the pivots, and the butterfly additions of up to 16
// columns' sums share their instructions (after the step of distance 16 a half-warp
// holds one column's partials, ...).  Then the triangle, a column per lane.
template <typename T>
__device__ __forceinline__ void bwd_front(const CtaFront& m, int row, const T* Bf, T* w, T* xp) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, c = m.c, f = m.f;
  T* X = w + m.woff;
  if (c < f) {
    const bool in = lane < f - c;
    const T x = in ? xp[row] : (T)0;
    const bool h = (lane & 16) != 0, g = (lane & 8) != 0, p = (lane & 4) != 0, o = (lane & 2) != 0;
    const T* B = Bf + c + (in ? lane : 0);
    for (int k0 = 0; k0 < c;) {
      T v;
      int k;
      if (c - k0 <= 4) {
        T a[4], b[2];
#pragma unroll
        for (int u = 0; u < 4; ++u) a[u] = (k0 + u < c) ? B[(k0 + u) * f] * x : (T)0;
#pragma unroll
        for (int t = 0; t < 2; ++t)
          b[t] = (h ? a[2 * t + 1] : a[2 * t]) + __shfl_xor_sync(FULL, h ? a[2 * t] : a[2 * t + 1], 16);
        v = (g ? b[1] : b[0]) + __shfl_xor_sync(FULL, g ? b[0] : b[1], 8);
        v += __shfl_xor_sync(FULL, v, 4);
        v += __shfl_xor_sync(FULL, v, 2);
        v += __shfl_xor_sync(FULL, v, 1);
        k = k0 + (h ? 1 : 0) + (g ? 2 : 0);
        if ((lane & 7) != 0) k = c;
        k0 += 4;
      } else {
        T a[16], b[8], d[4], e[2];
#pragma unroll
        for (int u = 0; u < 16; ++u) a[u] = (k0 + u < c) ? B[(k0 + u) * f] * x : (T)0;
#pragma unroll
        for (int t = 0; t < 8; ++t)
          b[t] = (h ? a[2 * t + 1] : a[2 * t]) + __shfl_xor_sync(FULL, h ? a[2 * t] : a[2 * t + 1], 16);
#pragma unroll
        for (int t = 0; t < 4; ++t)
          d[t] = (g ? b[2 * t + 1] : b[2 * t]) + __shfl_xor_sync(FULL, g ? b[2 * t] : b[2 * t + 1], 8);
#pragma unroll
        for (int t = 0; t < 2; ++t)
          e[t] = (p ? d[2 * t + 1] : d[2 * t]) + __shfl_xor_sync(FULL, p ? d[2 * t] : d[2 * t + 1], 4);
        v = (o ? e[1] : e[0]) + __shfl_xor_sync(FULL, o ? e[0] : e[1], 2);
        v += __shfl_xor_sync(FULL, v, 1);
        k = k0 + (h ? 1 : 0) + (g ? 2 : 0) + (p ? 4 : 0) + (o ? 8 : 0);
        if (lane & 1) k = c;
        k0 += 16;
      }
      if (k < c) X[k] -= v;
    }
    __syncwarp();
  }
  T v = lane < c ? X[lane] : (T)0;
  for (int j1 = c; j1 > 0; j1 -= 8) {
    T u8[8], d[4];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int j = j1 - 1 - u;
      u8[u] = (j >= 0 && lane < j) ? Bf[j + lane * f] : (T)0;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) d[u] = j1 - 2 - 2 * u >= 0 ? Bf[(j1 - 1 - 2 * u) + (j1 - 2 - 2 * u) * f] : (T)0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = j1 - 1 - 2 * u;
      if (j < 0) break;
      const T xa = __shfl_sync(FULL, v, j), xb0 = __shfl_sync(FULL, v, j > 0 ? j - 1 : 0);
      v -= u8[2 * u] * xa;
      if (j > 0) {
        const T xb = xb0 - d[u] * xa;
        v -= u8[2 * u + 1] * xb;
      }
    }
  }
  if (lane < c) xp[m.pos + lane] = v;
}

// The sweeps of a front of more than 32 rows by a warp, in 32-column blocks, the sums of
// k_fwd_front and k_bwd_front (after the division by D); eight columns' entries are
// loaded ahead of the chain that uses them.  G: the front's columns.
template <typename T>
__device__ __noinline__ void fwd_wide(const CtaPlan& cp, const CtaFront& m, const T* G, T* w) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, c = m.c, f = m.f;
  for (int t = lane; t < m.npull; t += 32) {
    const CtaPull pl = cp.pull[m.pull0 + t];
    T acc = w[pl.tg];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (u < pl.n) acc += w[pl.s[u]];
    for (int q = 4; q < pl.n; q += 8) {
      T v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = q + u < pl.n ? w[cp.pl_src[pl.more + q + u - 4]] : (T)0;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (q + u < pl.n) acc += v[u];
    }
    w[pl.tg] = acc;
  }
  __syncwarp();
  T* wj = w + m.woff;
  for (int j0 = 0; j0 < c; j0 += 32) {
    const int jb = min(32, c - j0);
    T xi = (lane < jb) ? wj[j0 + lane] : (T)0;
    for (int b = 0; b < jb; b += 8) {
      T v[8], d[4];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = (b + u < jb && lane > b + u && lane < jb) ? G[(j0 + lane) + (j0 + b + u) * f] : (T)0;
#pragma unroll
      for (int u = 0; u < 4; ++u) d[u] = b + 2 * u + 1 < jb ? G[(j0 + b + 2 * u + 1) + (j0 + b + 2 * u) * f] : (T)0;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int j = b + 2 * u;
        if (j >= jb) break;
        const T xa = __shfl_sync(FULL, xi, j), xb0 = __shfl_sync(FULL, xi, (j + 1) & 31);
        xi -= v[2 * u] * xa;
        if (j + 1 < jb) {
          const T xb = xb0 - d[u] * xa;
          xi -= v[2 * u + 1] * xb;
        }
      }
    }
    if (lane < jb) wj[j0 + lane] = xi;
    __syncwarp();
    for (int i = j0 + jb + lane; i < f; i += 32) {
      T s = (T)0;
#pragma unroll 8
      for (int jj = 0; jj < jb; ++jj) s += G[i + (j0 + jj) * f] * wj[j0 + jj];
      wj[i] -= s;
    }
    __syncwarp();
  }
}
template <typename T>
__device__ __noinline__ void bwd_wide(const CtaPlan& cp, const CtaFront& m, const T* G, T* w, T* xp) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, c = m.c, f = m.f;
  T* X = w + m.woff;
  for (int i = c + lane; i < f; i += 32) X[i] = xp[cp.rows_loc[m.rows + i - c]];
  __syncwarp();
  for (int j1 = c; j1 > 0; j1 -= 32) {
    const int j0 = max(0, j1 - 32);
    if (j1 < f)
      for (int k0 = j0; k0 < j1; k0 += 4) {
        T a[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) a[u] = (T)0;
        for (int i = j1 + lane; i < f; i += 32) {
          const T x = X[i];
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (k0 + u < j1) a[u] += G[i + (k0 + u) * f] * x;
        }
        const bool h = (lane & 16) != 0, g = (lane & 8) != 0;
        const T b0 = (h ? a[1] : a[0]) + __shfl_xor_sync(FULL, h ? a[0] : a[1], 16);
        const T b1 = (h ? a[3] : a[2]) + __shfl_xor_sync(FULL, h ? a[2] : a[3], 16);
        T v = (g ? b1 : b0) + __shfl_xor_sync(FULL, g ? b0 : b1, 8);
        v += __shfl_xor_sync(FULL, v, 4);
        v += __shfl_xor_sync(FULL, v, 2);
        v += __shfl_xor_sync(FULL, v, 1);
        const int k = k0 + (h ? 1 : 0) + (g ? 2 : 0);
        if ((lane & 7) == 0 && k < j1) X[k] -= v;
      }
    __syncwarp();
    const int jb = j1 - j0;
    T vi = (lane < jb) ? X[j0 + lane] : (T)0;
    for (int b = jb; b > 0; b -= 8) {
      T v[8], d[4];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = (b - 1 - u >= 0 && lane < b - 1 - u) ? G[(j0 + b - 1 - u) + (j0 + lane) * f] : (T)0;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        d[u] = b - 2 - 2 * u >= 0 ? G[(j0 + b - 1 - 2 * u) + (j0 + b - 2 - 2 * u) * f] : (T)0;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int j = b - 1 - 2 * u;
        if (j < 0) break;
        const T xa = __shfl_sync(FULL, vi, j), xb0 = __shfl_sync(FULL, vi, j > 0 ? j - 1 : 0);
        vi -= v[2 * u] * xa;
        if (j > 0) {
          const T xb = xb0 - d[u] * xa;
          vi -= v[2 * u + 1] * xb;
        }
      }
    }
    if (lane < jb) {
      X[j0 + lane] = vi;
      xp[m.pos + j0 + lane] = vi;
    }
    __syncwarp();
  }
}

// rhs norm, solve, residual, refinement test, until the test ends the refinement: the
// steps of Solver::kkt_solve for one problem.  kCtaSweepWarps warps sweep; a warp's next
// front (its columns by cp.async into the warp's other buffer, its pull list or update
// rows into registers, the descriptor after it) is on its way while the current one is
// processed, so that a level costs shared-memory accesses and the front's pivots only.
// All warps take part in the residual.
template <typename T>
__global__ void __launch_bounds__(kCtaThreads, 1)
    k_kkt_cta(CtaPlan cp, KmvArgs km, const T* __restrict__ F, const T* __restrict__ Dp, CtaRhs ra, CtaRhs rb,
              IterScal* sc, IrParams ir, const int* skip) {
  if (skip && *skip) return;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ unsigned long long s_max;
  __shared__ int s_go, s_rev;
  __shared__ IrState q;
  const CtaProblem pr = cp.prob[blockIdx.x];
  if (sc[blockIdx.x].halt) return;
  const double* __restrict__ rhs = blockIdx.y ? rb.rhs : ra.rhs;
  double* sol = blockIdx.y ? rb.sol : ra.sol;
  double* rr = blockIdx.y ? rb.r : ra.r;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  T* buf = reinterpret_cast<T*>(smraw) + (size_t)(wid < kCtaSweepWarps ? wid : 0) * 2 * cp.max_cols;
  T* const wide = reinterpret_cast<T*>(smraw) + (size_t)kCtaSweepWarps * 2 * cp.max_cols;
  T* w = wide + cp.max_wide;
  T* xp = w + pr.wtot;
  int32_t* lp = reinterpret_cast<int32_t*>(xp + pr.N);
  const int32_t* perm = cp.perm + pr.pos0;
  const T* D = Dp + pr.pos0;
  for (int l = tid; l <= pr.nlev; l += kCtaThreads) lp[l] = cp.lev_ptr[pr.lev0 + l];
  if (tid == 0) s_max = 0ull;
  if (pr.wide >= 0) {  // stays in shared memory for every sweep
    const CtaFront e = cp.front[pr.wide];
    for (int k = tid; k < e.c * e.f; k += kCtaThreads) wide[k] = F[e.goff + k];
  }
  __syncthreads();
  {
    double mx = 0.0;
    for (int k = tid; k < pr.N; k += kCtaThreads) {
      const double a = fabs(rhs[perm[k]]);
      mx = (a == a) ? fmax(mx, a) : INFINITY;  // a NaN entry makes the norm infinite
    }
    mx = warp_max(mx);
    if (lane == 0) atomicMax(&s_max, dbits(mx));
  }
  __syncthreads();
  if (tid == 0) {
    q = IrState{};
    q.rhs_norm = bitsd(s_max);
    q.ir_prev = INFINITY;
  }
  const bool sweep = wid < kCtaSweepWarps;
  auto staged = [](const CtaFront& e) { return e.c * e.f <= kCtaStage; };
  const double* b = rhs;
  for (bool add = false;; add = true, b = rr) {
    for (int t = tid; t < pr.wtot; t += kCtaThreads) {
      const int i = cp.w_init[pr.w0 + t];
      w[t] = (i >= 0) ? (T)b[i] : (T)0;
    }
    __syncthreads();
    if (sweep) {
      FrontSeq it(lp, pr.nlev, 1, wid);
      CtaFront m{}, mn{};
      CtaPull pc{}, pn{};
      auto pull_of = [&](const CtaFront& e) { return lane < e.npull ? cp.pull[e.pull0 + lane] : CtaPull{}; };
      int par = 0, cur = it.l;  // level of m
      if (!it.done()) {
        m = cp.front[it.j];
        if (staged(m)) warp_copy_async(buf, F + m.goff, m.c * m.f);
        pc = pull_of(m);
      }
      cp_commit();
      bool have = !it.done();
      it.next();
      int lev_n = it.l;
      bool have_n = !it.done();
      if (have_n) mn = cp.front[it.j];
      for (int l = 0; l < pr.nlev; ++l) {
        while (have && cur == l) {
          __syncwarp();  // every lane is done with the other buffer
          if (have_n) {
            if (staged(mn)) warp_copy_async(buf + (par ^ 1) * cp.max_cols, F + mn.goff, mn.c * mn.f);
            pn = pull_of(mn);
          }
          cp_commit();
          it.next();
          CtaFront m2{};
          const bool have2 = have_n && !it.done();
          if (have2) m2 = cp.front[it.j];
          cp_wait1();
          __syncwarp();
          const T* cols = staged(m) ? buf + par * cp.max_cols : wide;
          if (m.f <= 32) fwd_front<T>(cp, m, pc, cols, w);
          else fwd_wide<T>(cp, m, cols, w);
          m = mn;
          pc = pn;
          have = have_n;
          cur = lev_n;
          mn = m2;
          have_n = have2;
          lev_n = it.l;
          par ^= 1;
        }
        asm volatile("barrier.sync 1, %0;" ::"n"(32 * kCtaSweepWarps) : "memory");
      }
    }
    __syncthreads();
    // y / D of every pivot at once (a division per front and level would wait 569 clocks each)
    for (int k = tid; k < pr.N; k += kCtaThreads) {
      const int t = cp.slot[pr.pos0 + k];
      w[t] = w[t] / D[k];
    }
    __syncthreads();
    if (sweep) {
      FrontSeq it(lp, pr.nlev, -1, wid);
      CtaFront m{}, mn{};
      int par = 0, cur = it.l, rc = 0, rn = 0;
      auto row_of = [&](const CtaFront& e) { return lane < e.f - e.c ? cp.rows_loc[e.rows + lane] : 0; };
      if (!it.done()) {
        m = cp.front[it.j];
        if (staged(m)) warp_copy_async(buf, F + m.goff, m.c * m.f);
        rc = row_of(m);
      }
      cp_commit();
      bool have = !it.done();
      it.next();
      int lev_n = it.l;
      bool have_n = !it.done();
      if (have_n) mn = cp.front[it.j];
      for (int l = pr.nlev - 1; l >= 0; --l) {
        while (have && cur == l) {
          __syncwarp();  // every lane is done with the other buffer
          if (have_n) {
            if (staged(mn)) warp_copy_async(buf + (par ^ 1) * cp.max_cols, F + mn.goff, mn.c * mn.f);
            rn = row_of(mn);
          }
          cp_commit();
          it.next();
          CtaFront m2{};
          const bool have2 = have_n && !it.done();
          if (have2) m2 = cp.front[it.j];
          cp_wait1();
          __syncwarp();
          const T* cols = staged(m) ? buf + par * cp.max_cols : wide;
          if (m.f <= 32) bwd_front<T>(m, rc, cols, w, xp);
          else bwd_wide<T>(cp, m, cols, w, xp);
          m = mn;
          rc = rn;
          have = have_n;
          cur = lev_n;
          mn = m2;
          have_n = have2;
          lev_n = it.l;
          par ^= 1;
        }
        asm volatile("barrier.sync 1, %0;" ::"n"(32 * kCtaSweepWarps) : "memory");
      }
    }
    __syncthreads();
    for (int k = tid; k < pr.N; k += kCtaThreads) {
      const int i = perm[k];
      sol[i] = add ? sol[i] + (double)xp[k] : (double)xp[k];
    }
    if (tid == 0) s_max = 0ull;
    __syncthreads();
    {
      unsigned long long mx = 0ull;
      const int4* kr = km.krow + pr.pos0;
      const int32_t* ke = km.kcls + (int64_t)kKrowClasses * blockIdx.x;
      auto put = [&](int i, double x, double y) {
        const double r = rhs[i] - (x + y);
        rr[i] = r;
        const unsigned long long bt = dbits(fabs(r));
        mx = bt > mx ? bt : mx;
      };
      // the short rows a thread each (a warp holds one length class), the longest class first
      auto rows = [&](auto m_, int cls) {
        constexpr int M = decltype(m_)::value;
        for (int k = (cls ? ke[cls - 1] : 0) + tid; k < ke[cls]; k += kCtaThreads) {
          const int4 e = kr[k];
          double x, y;
          kmv_row_thread<M>(e.x, e.y, e.z, km.n, km.kcol, km.kvi, km.kval, km.kfv, sol, x, y);
          put(e.x, x, y);
        }
      };
      rows(std::integral_constant<int, 32>{}, 5);
      rows(std::integral_constant<int, 16>{}, 4);
      rows(std::integral_constant<int, 8>{}, 3);
      rows(std::integral_constant<int, 4>{}, 2);
      rows(std::integral_constant<int, 2>{}, 1);
      rows(std::integral_constant<int, 1>{}, 0);
      for (int k = ke[kKrowClasses - 2] + wid; k < ke[kKrowClasses - 1]; k += kCtaThreads / 32) {
        const int4 e = kr[k];
        double x, y;
        kmv_row<32>(e.x, e.y, e.z, km.n, km.kcol, km.kvi, km.kval, km.kfv, sol, lane, 0xffffffffu, x, y);
        if (lane == 0) put(e.x, x, y);
      }
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long t = __shfl_xor_sync(0xffffffffu, mx, o);
        mx = t > mx ? t : mx;
      }
      if (lane == 0) atomicMax(&s_max, mx);
    }
    __syncthreads();
    if (tid == 0) {
      q.rnorm_bits = s_max;
      s_go = ir_step_due(q, ir.abstol, ir.reltol, ir.stop_ratio, ir.max_steps) ? 1 : 0;
      s_rev = q.ir_revert;
    }
    __syncthreads();
    if (s_rev)
      for (int k = tid; k < pr.N; k += kCtaThreads) sol[perm[k]] -= (double)xp[k];
    if (!s_go) break;
  }
  // (sums and maxima: the same whichever right-hand side of the problem ends first)
  if (tid == 0) {
    IterScal& o = sc[blockIdx.x];
    atomicAdd(&o.ir_total, q.ir_total);
    if (q.ir_fail) atomicMax(&o.ir_fail, q.ir_fail);
    if (q.ir_worst > 0) atomicMax(reinterpret_cast<unsigned long long*>(&o.ir_worst), dbits(q.ir_worst));
  }
}

// Extend-add and partial LDL^T of every front of a problem, level by level, the
// operations of k_pull and k_factor_small: a warp per front, or four where a level has
// few fronts (the pivots are a serial chain: reciprocal 354 clocks, then the entries'
// two FP64 instructions at 64 clocks each, a quarter as many with four warps).
template <typename T>
__global__ void __launch_bounds__(kCtaThreads, 1)
    k_factor_cta(CtaPlan cp, T* F, T* __restrict__ Dp, const int8_t* __restrict__ dsign,
                 const int64_t* __restrict__ fa_tgt, const int64_t* __restrict__ fa_ptr,
                 const int64_t* __restrict__ fa_src, double eps_d, double delta_d, int* hits, const int* skip) {
  if (skip && *skip) return;
  extern __shared__ __align__(16) unsigned char smraw[];
  const CtaProblem pr = cp.prob[blockIdx.x];
  const int tid = threadIdx.x, wid = tid >> 5;
  constexpr int NW = kCtaThreads / 32;
  const int fw = cp.max_front;
  T* S0 = reinterpret_cast<T*>(smraw);
  const T eps = (T)eps_d, delta = (T)delta_d;
  // load of a front into S (f x f) and its extend-add in list order, by threads t0, t0 + nt, ...
  auto load = [&](T* S, const CtaFront& m, int t0, int nt) {
    const T* G = F + m.goff;
    for (int q = t0; q < m.f * m.f; q += nt) S[q] = G[q];
  };
  auto pull = [&](T* S, const CtaFront& m, int t0, int nt) {
    for (int64_t t = m.fa0 + t0; t < m.fa0 + m.nfa; t += nt) {
      const int64_t q1 = fa_ptr[t + 1];
      T* s = S + (fa_tgt[t] - m.goff);
      T acc = *s;
      for (int64_t q = fa_ptr[t]; q < q1; ++q) acc += F[fa_src[q]];
      *s = acc;
    }
  };
  const int32_t* lp = cp.lev_ptr + pr.lev0;
  for (int l = 0; l < pr.nlev; ++l) {
    const int j0 = lp[l], j1 = lp[l + 1];
    if (j1 - j0 > NW / 4) {
      for (int j = j0 + wid; j < j1; j += NW) {
        const CtaFront m = cp.front[j];
        T* S = S0 + wid * front_words(fw);
        load(S, m, tid & 31, 32);
        __syncwarp();
        pull(S, m, tid & 31, 32);
        factor_front32<T, 1>(S, F + m.goff, Dp + pr.pos0 + m.pos, dsign + pr.pos0 + m.pos, m.c, m.f, eps, delta, hits, 0);
      }
    } else if (j0 + wid / 4 < j1) {
      const CtaFront m = cp.front[j0 + wid / 4];
      const int bar = 1 + wid / 4;
      T* S = S0 + (wid / 4) * front_words(fw);
      load(S, m, tid & 127, 128);
      asm volatile("barrier.sync %0, 128;" ::"r"(bar) : "memory");
      pull(S, m, tid & 127, 128);
      factor_front32<T, 4>(S, F + m.goff, Dp + pr.pos0 + m.pos, dsign + pr.pos0 + m.pos, m.c, m.f, eps, delta, hits, bar);
    }
    __syncthreads();
  }
}

size_t factor_smem(const CtaPlan& cp, size_t word) {
  return word * (size_t)(kCtaThreads / 32) * (size_t)front_words(cp.max_front);
}
size_t solve_smem(const CtaPlan& cp, size_t word) {
  return word * ((size_t)cp.max_slots + (size_t)cp.max_wide + 2 * (size_t)kCtaSweepWarps * (size_t)cp.max_cols) +
         sizeof(int32_t) * (size_t)(cp.max_levels + 1);
}

}  // namespace

// Times of a set of CTAs on the GPU: the longest, or, with more than one per SM, the list schedule's bound.
static double cta_makespan(const std::vector<double>& t, int copies) {
  double sum = 0.0, most = 0.0;
  for (double x : t) sum += x, most = std::max(most, x);
  return copies * (int64_t)t.size() <= kSMs ? most : copies * sum / kSMs + most * (1.0 - 1.0 / kSMs);
}

static CtaCost cta_cost(const Symbolic& sy, const std::vector<std::vector<std::pair<int32_t, int64_t>>>& byp) {
  CtaCost k;
  std::vector<double> solve(sy.nlev, 0.0), fac(sy.nlev, 0.0), pf;  // by launches: the longest front of a level
  for (const auto& fronts : byp) {
    double t = 16.0, tf = 8.0;
    for (size_t i = 0; i < fronts.size();) {
      const int32_t l = fronts[i].first;
      size_t j = i;
      while (j < fronts.size() && fronts[j].first == l) ++j;
      double w8[kCtaSweepWarps] = {}, w16[kCtaThreads / 32] = {}, four = 0.0;
      for (size_t q = i; q < j; ++q) {
        const int64_t J = fronts[q].second;
        const double c = (double)(sy.sn_ptr[J + 1] - sy.sn_ptr[J]), f = (double)(sy.row_ptr[J + 1] - sy.row_ptr[J]);
        const double by4 = 0.55 * c + 1.6e-4 * c * f * f;  // four warps: the chain of pivots, then the entries
        w8[(q - i) % kCtaSweepWarps] += 0.9 + 0.2 * c + (f > 32 ? 0.005 * c * f : 0.0);
        w16[(q - i) % (kCtaThreads / 32)] += 2.1 + 0.55 * c + 1e-3 * c * f * f;
        four = std::max(four, 1.5 + by4);
        solve[l] = std::max(solve[l], 0.25 * c + 0.003 * c * f);
        fac[l] = std::max(fac[l], by4);
      }
      t += 0.4 + *std::max_element(w8, w8 + kCtaSweepWarps);
      tf += j - i <= 4 ? four : 1.0 + *std::max_element(w16, w16 + kCtaThreads / 32);
      i = j;
    }
    k.sweep.push_back(t);
    pf.push_back(tf);
  }
  k.levels = 21.0 + 1.6e-3 * (double)sy.N;
  k.factor_levels = 7.0 + 2e-3 * (double)sy.nsn;
  for (int64_t l = 0; l < sy.nlev; ++l) {
    k.levels += 5.5 + solve[l];
    k.factor_levels += 4.5 + fac[l];
  }
  k.factor = cta_makespan(pf, 1);
  return k;
}

bool cta_solve_pays(const CtaCost& c, const std::vector<int64_t>& entries) {
  std::vector<double> t(c.sweep);
  double all = 0.0;
  for (size_t p = 0; p < t.size(); ++p) {
    t[p] += 3.5e-3 * (double)entries[p];
    all += (double)entries[p];
  }
  // (6 %: the initial point's two right-hand sides share a launch too)
  return cta_makespan(t, 2) + cta_makespan(t, 1) < 1.06 * 3.0 * (c.levels + 6e-5 * all);
}

int cta_plan_build(DeviceArena& ar, const Symbolic& sy, const NumericMaps& mp, int small_max,
                   const std::vector<int32_t>* pos_pid, const int32_t* d_w_init, CtaPlan& out, CtaCost& cost) {
  out = CtaPlan();
  cost = CtaCost();
  if (sy.nsn == 0 || sy.max_front > std::min(small_max, kCtaRows) || sy.N >= ((int64_t)1 << 31) || sy.upd_total >= ((int64_t)1 << 31))
    return CLR_OK;
  auto pid_of = [&](int64_t J) { return pos_pid ? (*pos_pid)[sy.sn_ptr[J]] : 0; };
  int64_t B = 1;
  for (int64_t J = 0; J < sy.nsn; ++J) B = std::max<int64_t>(B, pid_of(J) + 1);
  // problems hold contiguous runs of supernodes, positions and solve slots, in order
  std::vector<CtaProblem> pb(B);
  std::vector<int64_t> work(B, 0), j0(B, -1), nwide(B, 0);
  for (int64_t J = 0; J < sy.nsn; ++J) {
    const int64_t p = pid_of(J), c = sy.sn_ptr[J + 1] - sy.sn_ptr[J], f = sy.row_ptr[J + 1] - sy.row_ptr[J];
    if (j0[p] < 0) {
      j0[p] = J;
      pb[p].pos0 = (int32_t)sy.sn_ptr[J];
      pb[p].w0 = sy.upd_off[J];
    } else if (pid_of(J - 1) != p || sy.upd_off[J] != sy.upd_off[J - 1] + (sy.row_ptr[J] - sy.row_ptr[J - 1])) {
      return CLR_OK;  // (not laid out as assumed: the general path)
    }
    pb[p].N += (int32_t)c;
    pb[p].wtot += (int32_t)f;
    work[p] += c * f;
    if (c * f <= kCtaStage) {
      out.max_cols = std::max(out.max_cols, (int32_t)(c * f));
    } else {
      out.max_wide = std::max(out.max_wide, (int32_t)(c * f));
      ++nwide[p];
    }
  }
  for (int64_t p = 0; p < B; ++p) {
    if (j0[p] < 0 || work[p] > kCtaWork || nwide[p] > 1) return CLR_OK;
    if (p > 0 && pb[p].pos0 <= pb[p - 1].pos0) return CLR_OK;  // (problems in elimination order)
    out.max_slots = std::max(out.max_slots, pb[p].N + pb[p].wtot);
  }
  out.max_levels = (int32_t)sy.nlev;
  out.max_front = (int32_t)sy.max_front;
  out.factor = out.max_front <= kCtaWarpRows;
  if (solve_smem(out, 8) > (size_t)kCtaSmem) return CLR_OK;
  if (!mp.px_child.empty()) out.factor = false;  // children pushed by relative indices: the general path
  std::vector<std::vector<std::pair<int32_t, int64_t>>> byp(B);  // (level, front) of each problem, level-major
  for (int64_t l = 0; l < sy.nlev; ++l)
    for (int64_t t = sy.lev_ptr[l]; t < sy.lev_ptr[l + 1]; ++t) byp[pid_of(sy.lev_sn[t])].emplace_back((int32_t)l, sy.lev_sn[t]);
  // pull targets of each front: they come level by level, front by front, in order
  std::vector<int64_t> sv0(sy.nsn, 0), sv1(sy.nsn, 0), fa0(sy.nsn, 0), fa1(sy.nsn, 0);
  for (int64_t l = 0; l < sy.nlev; ++l) {
    int64_t t = mp.sv_lev_ptr[l], a = mp.fa_lev_ptr[l];
    for (int64_t k = sy.lev_ptr[l]; k < sy.lev_ptr[l + 1]; ++k) {
      const int64_t J = sy.lev_sn[k], f = sy.row_ptr[J + 1] - sy.row_ptr[J];
      sv0[J] = t;
      while (t < mp.sv_lev_ptr[l + 1] && mp.sv_tgt[t] >= sy.upd_off[J] && mp.sv_tgt[t] < sy.upd_off[J] + f) ++t;
      sv1[J] = t;
      fa0[J] = a;
      while (a < mp.fa_lev_ptr[l + 1] && mp.fa_tgt[a] >= sy.front_off[J] && mp.fa_tgt[a] < sy.front_off[J] + f * f) ++a;
      fa1[J] = a;
    }
    if (t != mp.sv_lev_ptr[l + 1] || a != mp.fa_lev_ptr[l + 1]) return CLR_OK;
  }
  cost = cta_cost(sy, byp);
  if (!(cost.factor < 0.9 * cost.factor_levels)) out.factor = false;
  std::vector<CtaFront> fr;
  std::vector<CtaPull> pulls;
  std::vector<int32_t> lev, rows, psrc, perm(sy.N), slot(sy.N);
  for (int64_t k = 0; k < sy.N; ++k) perm[k] = (int32_t)sy.perm[k];
  for (int64_t p = 0; p < B; ++p) {
    pb[p].lev0 = (int32_t)lev.size();
    pb[p].wide = -1;
    int32_t cur = -1;
    for (const auto& [l, J] : byp[p]) {
      const int64_t c = sy.sn_ptr[J + 1] - sy.sn_ptr[J], f = sy.row_ptr[J + 1] - sy.row_ptr[J];
      if (l != cur) {  // (levels without fronts of this problem do not occur: a parent is one level up or more)
        cur = l;
        lev.push_back((int32_t)fr.size());
        ++pb[p].nlev;
      }
      CtaFront m{};
      m.goff = sy.front_off[J];
      m.c = (int32_t)c;
      m.f = (int32_t)f;
      m.woff = (int32_t)(sy.upd_off[J] - pb[p].w0);
      m.pos = (int32_t)(sy.sn_ptr[J] - pb[p].pos0);
      m.rows = (int32_t)rows.size();
      for (int64_t k = 0; k < c; ++k) slot[sy.sn_ptr[J] + k] = (int32_t)(m.woff + k);
      for (int64_t a = c; a < f; ++a) rows.push_back((int32_t)(sy.rows[sy.row_ptr[J] + a] - pb[p].pos0));
      m.pull0 = (int32_t)pulls.size();
      m.npull = (int32_t)(sv1[J] - sv0[J]);
      for (int64_t t = sv0[J]; t < sv1[J]; ++t) {
        const int64_t n = mp.sv_ptr[t + 1] - mp.sv_ptr[t];
        if (n > kPullSerial) return CLR_OK;  // (not summed in list order there)
        CtaPull e{};
        e.tg = (uint16_t)(mp.sv_tgt[t] - pb[p].w0);
        e.n = (uint16_t)n;
        e.more = (int32_t)psrc.size();
        for (int64_t q = 0; q < n; ++q) {
          const int64_t sl = mp.sv_src[mp.sv_ptr[t] + q] - pb[p].w0;
          if (q < 4) e.s[q] = (uint16_t)sl;
          else psrc.push_back((int32_t)sl);
        }
        pulls.push_back(e);
      }
      m.fa0 = fa0[J];
      m.nfa = (int32_t)(fa1[J] - fa0[J]);
      for (int64_t t = fa0[J]; t < fa1[J]; ++t)
        if (mp.fa_ptr[t + 1] - mp.fa_ptr[t] > kPullSerial) out.factor = false;
      if (c * f > kCtaStage) pb[p].wide = (int32_t)fr.size();
      fr.push_back(m);
    }
    lev.push_back((int32_t)fr.size());  // end of the problem's last level
  }
  out.prob = ar.upload(pb.data(), B);
  out.front = ar.upload(fr.data(), (int64_t)fr.size());
  out.lev_ptr = ar.upload(lev.data(), (int64_t)lev.size());
  out.rows_loc = ar.upload(rows.data(), (int64_t)rows.size());
  out.pull = ar.upload(pulls.data(), (int64_t)pulls.size());
  out.pl_src = ar.upload(psrc.data(), (int64_t)psrc.size());
  out.perm = ar.upload(perm.data(), sy.N);
  out.slot = ar.upload(slot.data(), sy.N);
  out.w_init = d_w_init;
  if (!out.prob || !out.front || !out.lev_ptr || !out.rows_loc || !out.pull || !out.pl_src || !out.perm || !out.slot)
    return CLR_E_OOM;
  out.n = B;
  return CLR_OK;
}

template <typename T>
int CtaOps<T>::setup_attributes() {
  CLR_CUDA(cudaFuncSetAttribute(k_kkt_cta<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCtaSmem));
  CLR_CUDA(cudaFuncSetAttribute(k_factor_cta<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCtaSmem));
  return CLR_OK;
}

template <typename T>
int CtaOps<T>::factor(cudaStream_t st, const CtaPlan& cp, T* F, T* Dp, const int8_t* dsign, const int64_t* fa_tgt,
                      const int64_t* fa_ptr, const int64_t* fa_src, double eps, double delta, int* hits,
                      const int* skip) {
  k_factor_cta<T><<<(unsigned)cp.n, kCtaThreads, factor_smem(cp, sizeof(T)), st>>>(cp, F, Dp, dsign, fa_tgt, fa_ptr,
                                                                                   fa_src, eps, delta, hits, skip);
  CLR_CHECK_LAUNCH();
  return CLR_OK;
}

template <typename T>
int CtaOps<T>::kkt_solve(cudaStream_t st, const CtaPlan& cp, const KmvArgs& k, const T* F, const T* Dp,
                         const CtaRhs& a, const CtaRhs& b, IterScal* sc, const IrParams& ir, const int* skip) {
  k_kkt_cta<T><<<dim3((unsigned)cp.n, b.rhs ? 2u : 1u), kCtaThreads, solve_smem(cp, sizeof(T)), st>>>(cp, k, F, Dp, a, b,
                                                                                                 sc, ir, skip);
  CLR_CHECK_LAUNCH();
  return CLR_OK;
}

template struct CtaOps<double>;
template struct CtaOps<float>;

}  // namespace clr
