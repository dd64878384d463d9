// Many thin leaf fronts of one parent: their extend-add as one product, their solves by columns.
//
// A parent with hundreds of thin leaves (a portfolio: one leaf per asset with its row of the
// factor matrix) sums their update matrices l d l^T entry by entry: r^2 / 2 values written by every
// leaf, and for every one of them an index and a gathered value read, a sector of 32 bytes each
// when the leaves' rows are random subsets (n = 5000, 500 factors half dense: 1.6e8 values, 1.22 ms
// of gathers, 0.2 ms of stores and 0.19 ms to clear their 1.25 GB of the pool per factorization).
// The sum is W^T D W with W the leaves' columns scattered into the parent's rows, 10 MB: the zeros cost
// FMAs (6.3e8 here, of which a quarter count) and no memory: 124 us with the clearing, and 14 us in
// place of 209 for the leaves, which keep their columns only.
//
// Tiles of 64 x 64 of the lower triangle, 4 x 4 per thread, the columns in splits so that small
// parents fill the SMs (about 608 CTAs: four per SM); partial tiles are added in the order of
// the splits, which depend on the parent alone.
//
// Solves: w_P -= W^T y over the panel (coalesced, L2 resident) in place of a CTA per leaf and 5000
// sources gathered per entry of w_P (13.5 + 11.4 us), and a warp per leaf for its columns' dot
// products with the ancestors (a CTA of 256 threads with four barriers each took 24 us): 21 us together, launches included.
#include "thinsyrk.cuh"

#include <algorithm>

namespace clr {
namespace {
constexpr int TB = 64, TK = 16, NT = 256;
constexpr int64_t kCtas = 608, kSegment = 1 << 15;

template <typename T>
__global__ void k_clear_segments(T* __restrict__ F, const int64_t* __restrict__ seg) {
  const int64_t o = seg[2 * blockIdx.x], n = seg[2 * blockIdx.x + 1];
  for (int64_t k = threadIdx.x; k < n; k += blockDim.x) F[o + k] = (T)0;
}

// a warp per column; W's zeros never change
template <typename T>
__global__ void __launch_bounds__(NT) k_scatter_columns(const T* __restrict__ F, T* __restrict__ W, ThinSyrkParent p,
                                                        const int64_t* __restrict__ src, const int64_t* __restrict__ map0,
                                                        const int32_t* __restrict__ cnt, const int32_t* __restrict__ map,
                                                        const int* skip) {
  if (skip && *skip) return;
  const int64_t k = (blockIdx.x * (int64_t)NT + threadIdx.x) / 32;
  if (k >= p.K) return;
  const int64_t s = src[p.col0 + k];
  const int32_t* m = map + map0[p.col0 + k];
  const int n = cnt[p.col0 + k];
  T* w = W + p.woff + k * p.ld;
  for (int a = threadIdx.x & 31; a < n; a += 32) w[m[a]] = F[s + a];
}

template <typename T>
struct alignas(16) Vec4 {
  T v[4];
};

// Tile blockIdx.x (I >= J by rows of the triangle), split blockIdx.y.
template <typename T>
__global__ void __launch_bounds__(NT) k_syrk_tiles(T* __restrict__ F, const T* __restrict__ Dp,
                                                   const T* __restrict__ Wall, ThinSyrkParent p,
                                                   const int32_t* __restrict__ dpos, T* __restrict__ part,
                                                   const int* skip) {
  if (skip && *skip) return;
  __shared__ Vec4<T> As[2][TK][TB / 4], Bs[2][TK][TB / 4];
  int I = (int)((sqrtf(8.0f * (float)blockIdx.x + 1.0f) - 1.0f) * 0.5f);
  while ((int64_t)I * (I + 1) / 2 > blockIdx.x) --I;
  while ((int64_t)(I + 1) * (I + 2) / 2 <= blockIdx.x) ++I;
  const int J = (int)(blockIdx.x - (int64_t)I * (I + 1) / 2);
  const int64_t k0 = blockIdx.y * p.kc, k1 = min(p.K, k0 + p.kc);
  const int tid = threadIdx.x, kk = tid >> 4, q = tid & 15;  // loads: column kk of a step, rows 4 q ..
  const int tx = tid & 15, ty = tid >> 4;                   // product: rows 4 tx .., columns 4 ty ..
  const T* W = Wall + p.woff;
  Vec4<T> a, b;
  auto load = [&](int64_t k) {
    if (k < k1) {
      a = *reinterpret_cast<const Vec4<T>*>(W + k * p.ld + TB * I + 4 * q);
      b = *reinterpret_cast<const Vec4<T>*>(W + k * p.ld + TB * J + 4 * q);
      const T d = Dp[dpos[p.col0 + k]];
      // (an infinite pivot has l = 0 and takes nothing off, as in k_factor_thin: no 0 times infinity)
#pragma unroll
      for (int u = 0; u < 4; ++u) b.v[u] = b.v[u] == (T)0 ? (T)0 : b.v[u] * d;
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u) a.v[u] = b.v[u] = (T)0;
    }
  };
  T acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = (T)0;
  load(k0 + kk);
  int buf = 0;
  for (int64_t k = k0; k < k1; k += TK, buf ^= 1) {
    As[buf][kk][q] = a;
    Bs[buf][kk][q] = b;
    __syncthreads();
    load(k + TK + kk);
#pragma unroll
    for (int m = 0; m < TK; ++m) {
      const Vec4<T> x = As[buf][m][tx], y = Bs[buf][m][ty];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] += x.v[i] * y.v[j];
    }
  }
  if (p.splits > 1) {
    T* o = part + ((int64_t)blockIdx.x * p.splits + blockIdx.y) * (TB * TB);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      Vec4<T> v;
#pragma unroll
      for (int i = 0; i < 4; ++i) v.v[i] = acc[i][j];
      *reinterpret_cast<Vec4<T>*>(o + (4 * ty + j) * TB + 4 * tx) = v;
    }
  } else {
    T* G = F + p.goff;
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int64_t r = TB * I + 4 * tx + i, c = TB * J + 4 * ty + j;
        if (r < p.fP && r >= c) G[r + c * p.fP] -= acc[i][j];
      }
  }
}

template <typename T>
__global__ void __launch_bounds__(NT) k_add_tiles(T* __restrict__ F, ThinSyrkParent p, const T* __restrict__ part,
                                                  const int* skip) {
  if (skip && *skip) return;
  const int64_t tile = blockIdx.x / (TB * TB / NT);
  const int e = (int)(blockIdx.x % (TB * TB / NT)) * NT + threadIdx.x;
  int I = (int)((sqrtf(8.0f * (float)tile + 1.0f) - 1.0f) * 0.5f);
  while ((int64_t)I * (I + 1) / 2 > tile) --I;
  while ((int64_t)(I + 1) * (I + 2) / 2 <= tile) ++I;
  const int J = (int)(tile - (int64_t)I * (I + 1) / 2);
  const int64_t r = TB * I + (e & (TB - 1)), c = TB * J + e / TB;
  if (r >= p.fP || r < c) return;
  const T* o = part + tile * p.splits * (TB * TB) + e;
  T s = (T)0;
#pragma unroll 8
  for (int64_t k = 0; k < p.splits; ++k) s += o[k * (TB * TB)];
  F[p.goff + r + c * p.fP] -= s;
}

// Leaves of several pivots: the unit lower solve of their diagonal block, a warp each (c <= 32).
template <typename T>
__global__ void __launch_bounds__(NT) k_leaf_fwd(const T* __restrict__ F, T* __restrict__ w, const int64_t* __restrict__ front,
                                                 int64_t n, const int64_t* __restrict__ sn_ptr,
                                                 const int64_t* __restrict__ row_ptr,
                                                 const int64_t* __restrict__ front_off,
                                                 const int64_t* __restrict__ upd_off, const int* skip) {
  if (skip && *skip) return;
  const int64_t t = (blockIdx.x * (int64_t)NT + threadIdx.x) / 32;
  if (t >= n) return;
  const int lane = threadIdx.x & 31;
  const int64_t J = front[t], f = row_ptr[J + 1] - row_ptr[J];
  const int c = (int)(sn_ptr[J + 1] - sn_ptr[J]);
  const T* G = F + front_off[J];
  T x = lane < c ? w[upd_off[J] + lane] : (T)0;
  for (int j = 0; j < c; ++j) {
    const T xj = __shfl_sync(0xffffffffu, x, j);
    if (lane > j && lane < c) x -= G[lane + j * f] * xj;
  }
  if (lane < c) w[upd_off[J] + lane] = x;
}

// Split blockIdx.y of w_P's product: rows 256 blockIdx.x .., a thread each.
template <typename T>
__global__ void __launch_bounds__(NT) k_panel_product(const T* __restrict__ Wall, const T* __restrict__ w, ThinSyrkParent p,
                                                      const int64_t* __restrict__ slot, T* __restrict__ part,
                                                      const int* skip) {
  if (skip && *skip) return;
  __shared__ T y[NT];
  const int64_t i = blockIdx.x * (int64_t)NT + threadIdx.x;
  const int64_t k0 = blockIdx.y * p.vc, k1 = min(p.K, k0 + p.vc);
  const T* W = Wall + p.woff + min(i, p.ld - 1);
  T a[4] = {(T)0, (T)0, (T)0, (T)0};
  for (int64_t b = k0; b < k1; b += NT) {
    const int m = (int)min((int64_t)NT, k1 - b);
    __syncthreads();
    if ((int)threadIdx.x < m) y[threadIdx.x] = w[slot[p.col0 + b + threadIdx.x]];
    __syncthreads();
    int k = 0;
    for (; k + 8 <= m; k += 8) {
      T x[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) x[u] = W[(b + k + u) * p.ld];
#pragma unroll
      for (int u = 0; u < 8; ++u) a[u & 3] += x[u] * y[k + u];
    }
    for (; k < m; ++k) a[0] += W[(b + k) * p.ld] * y[k];
  }
  if (i < p.fP) part[blockIdx.y * p.fP + i] = (a[0] + a[1]) + (a[2] + a[3]);
}
template <typename T>
__global__ void __launch_bounds__(NT) k_panel_add(T* __restrict__ w, ThinSyrkParent p, const T* __restrict__ part,
                                                  const int* skip) {
  if (skip && *skip) return;
  // eight lanes per row: lane g adds the splits g, g + 8, ...
  const int64_t i = (blockIdx.x * (int64_t)NT + threadIdx.x) / 8;
  const int g = threadIdx.x & 7;
  T s = (T)0;
  if (i < p.fP)
    for (int64_t k = g; k < p.vsplits; k += 8) s += part[k * p.fP + i];
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (g == 0 && i < p.fP) w[p.wslot + i] -= s;
}

// Backward sweep of a leaf by a warp: v = y / D - sum over the rows below of l x, then its diagonal block.
template <typename T>
__global__ void __launch_bounds__(NT) k_leaf_bwd(const T* __restrict__ F, const T* __restrict__ Dp,
                                                 const T* __restrict__ w, T* __restrict__ xs,
                                                 const int64_t* __restrict__ front, int64_t n,
                                                 const int64_t* __restrict__ sn_ptr, const int64_t* __restrict__ row_ptr,
                                                 const int64_t* __restrict__ front_off,
                                                 const int64_t* __restrict__ upd_off,
                                                 const int32_t* __restrict__ rows_kkt, const int* skip) {
  if (skip && *skip) return;
  const int64_t t = (blockIdx.x * (int64_t)NT + threadIdx.x) / 32;
  if (t >= n) return;
  const int lane = threadIdx.x & 31;
  const int64_t J = front[t];
  const int c = (int)(sn_ptr[J + 1] - sn_ptr[J]), f = (int)(row_ptr[J + 1] - row_ptr[J]);
  const T* G = F + front_off[J];
  const int32_t* rk = rows_kkt + row_ptr[J];
  T v = lane < c ? w[upd_off[J] + lane] / Dp[sn_ptr[J] + lane] : (T)0;
  for (int k = c - 1; k >= 0; --k) {
    const T* g = G + (int64_t)k * f;
    T s[4] = {(T)0, (T)0, (T)0, (T)0};
    for (int i0 = c; i0 < f; i0 += 128) {
      T l[4], x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + 32 * u + lane;
        l[u] = i < f ? g[i] : (T)0;
        x[u] = i < f ? xs[rk[i]] : (T)0;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) s[u] += l[u] * x[u];
    }
    const T d = warp_sum((s[0] + s[1]) + (s[2] + s[3]));
    if (lane == k) v -= d;
  }
  for (int k = c - 1; k >= 0; --k) {
    const T xk = __shfl_sync(0xffffffffu, v, k);
    if (lane < k) v -= G[k + (int64_t)lane * f] * xk;
  }
  if (lane < c) xs[rk[lane]] = v;
}
}  // namespace

// The parents: at least min_children thin leaves, and the product's FMAs not more than `ratio` per
// value of the update matrices that they replace.
int thin_syrk_plan(DeviceArena& ar, const Symbolic& sy, const NumericMaps& mp, const std::vector<char>& leaf, int64_t ratio,
                   int64_t min_children, ThinSyrk& out, FaLists& fa, FaLists& sv) {
  out.lev.assign(sy.nlev, {});
  std::vector<char> pushed(sy.nsn, 0);
  for (int64_t J : mp.px_child) pushed[J] = 1;
  auto rows = [&](int64_t J) { return sy.row_ptr[J + 1] - sy.row_ptr[J]; };
  auto pivots = [&](int64_t J) { return sy.sn_ptr[J + 1] - sy.sn_ptr[J]; };
  std::vector<int64_t> num(sy.nsn, 0), cols(sy.nsn, 0), ne(sy.nsn, 0);
  for (int64_t J = 0; J < sy.nsn; ++J) {
    const int64_t P = sy.sn_parent[J];
    if (P < 0 || !leaf[J] || pushed[J]) continue;
    const int64_t r = rows(J) - pivots(J);
    ++num[P];
    cols[P] += pivots(J);
    ne[P] += r * (r + 1) / 2;
  }
  std::vector<char> take(sy.nsn, 0);
  bool any = false;
  for (int64_t P = 0; P < sy.nsn; ++P)
    if (num[P] >= min_children && rows(P) * (rows(P) + 1) / 2 * cols[P] <= ratio * ne[P]) take[P] = 1, any = true;
  if (!any) return CLR_OK;
  out.child.assign(sy.nsn, 0);
  std::vector<std::vector<int64_t>> kids(sy.nsn);
  for (int64_t J = 0; J < sy.nsn; ++J)
    if (sy.sn_parent[J] >= 0 && take[sy.sn_parent[J]]) {
      kids[sy.sn_parent[J]].push_back(J);
      out.child[J] = leaf[J] && !pushed[J];
    }
  std::vector<int64_t> src, map0, slot, front;
  std::vector<int32_t> cnt, dpos, map, loc(sy.N, -1);
  std::vector<std::pair<int64_t, int64_t>> contrib;
  // the targets in [lo, hi) of level l, which follow one another from t on: copied to `o` or skipped
  auto pass = [](const std::vector<int64_t>& tgt, const std::vector<int64_t>& ptr, const std::vector<int64_t>& s,
                 int64_t& t, int64_t t1, int64_t lo, int64_t hi, bool keep, FaLists& o) {
    for (; t < t1 && tgt[t] >= lo && tgt[t] < hi; ++t) {
      if (!keep) continue;
      o.tgt.push_back(tgt[t]);
      o.ptr.push_back((int64_t)o.src.size());
      o.src.insert(o.src.end(), s.begin() + ptr[t], s.begin() + ptr[t + 1]);
    }
  };
  auto lists = [&](FaLists& o) {
    std::stable_sort(contrib.begin(), contrib.end(), [](auto& a, auto& b) { return a.first < b.first; });
    for (size_t k = 0; k < contrib.size(); ++k) {
      if (k == 0 || contrib[k].first != contrib[k - 1].first) {
        o.tgt.push_back(contrib[k].first);
        o.ptr.push_back((int64_t)o.src.size());
      }
      o.src.push_back(contrib[k].second);
    }
    contrib.clear();
  };
  fa = sv = FaLists();
  fa.lev_ptr.assign(1, 0);
  sv.lev_ptr.assign(1, 0);
  for (int64_t l = 0; l < sy.nlev; ++l) {
    int64_t ts = mp.sv_lev_ptr[l];
    const int64_t ts1 = mp.sv_lev_ptr[l + 1];
    int64_t t = mp.fa_lev_ptr[l];
    const int64_t t1 = mp.fa_lev_ptr[l + 1];
    for (int64_t x = sy.lev_ptr[l]; x < sy.lev_ptr[l + 1]; ++x) {
      const int64_t P = sy.lev_sn[x], fP = rows(P);
      pass(mp.fa_tgt, mp.fa_ptr, mp.fa_src, t, t1, sy.front_off[P], sy.front_off[P] + fP * fP, !take[P], fa);
      pass(mp.sv_tgt, mp.sv_ptr, mp.sv_src, ts, ts1, sy.upd_off[P], sy.upd_off[P] + fP, !take[P], sv);
      if (!take[P]) continue;
      const int64_t* rP = sy.rows.data() + sy.row_ptr[P];
      for (int64_t a = 0; a < fP; ++a) loc[rP[a]] = (int32_t)a;
      ThinSyrkParent p{};
      p.goff = sy.front_off[P];
      p.fP = fP;
      p.ld = (fP + TB - 1) / TB * TB;
      p.K = cols[P];
      p.col0 = (int64_t)src.size();
      p.woff = out.wtotal;
      p.wslot = sy.upd_off[P];
      p.front0 = (int64_t)front.size();
      for (int64_t J : kids[P]) {
        const int64_t f = rows(J), c = pivots(J);
        const int64_t* r = sy.rows.data() + sy.row_ptr[J];
        if (pushed[J]) continue;
        if (!out.child[J]) {  // stays with the lists
          for (int64_t b = c; b < f; ++b)
            for (int64_t a = b; a < f; ++a)
              contrib.emplace_back(p.goff + loc[r[a]] + loc[r[b]] * fP, sy.front_off[J] + a + b * f);
          continue;
        }
        for (int64_t b = 0; b < c; ++b) {
          src.push_back(sy.front_off[J] + c + b * f);
          map0.push_back((int64_t)map.size());
          cnt.push_back((int32_t)(f - c));
          dpos.push_back((int32_t)(sy.sn_ptr[J] + b));
          slot.push_back(sy.upd_off[J] + b);
        }
        front.push_back(J);
        p.many |= c > 1;
        for (int64_t a = c; a < f; ++a) map.push_back(loc[r[a]]);
      }
      lists(fa);
      for (int64_t J : kids[P]) {
        if (out.child[J]) continue;
        const int64_t* r = sy.rows.data() + sy.row_ptr[J];
        for (int64_t a = pivots(J); a < rows(J); ++a)
          contrib.emplace_back(sy.upd_off[P] + loc[r[a]], sy.upd_off[J] + a);
      }
      lists(sv);
      p.nfront = (int64_t)front.size() - p.front0;
      p.vc = std::max<int64_t>(32, (p.K * ((fP + NT - 1) / NT) + kCtas - 1) / kCtas);
      p.vsplits = (p.K + p.vc - 1) / p.vc;
      out.part = std::max(out.part, p.vsplits * fP);
      const int64_t nt = p.ld / TB;
      p.tiles = nt * (nt + 1) / 2;
      p.splits = std::max<int64_t>(1, std::min((kCtas + p.tiles - 1) / p.tiles, p.K / 64));
      p.kc = ((p.K + p.splits - 1) / p.splits + TK - 1) / TK * TK;
      p.splits = (p.K + p.kc - 1) / p.kc;
      if (p.splits > 1) out.part = std::max(out.part, p.tiles * p.splits * TB * TB);
      out.wtotal += p.K * p.ld;
      out.lev[l].push_back(p);
    }
    fa.lev_ptr.push_back((int64_t)fa.tgt.size());
    sv.lev_ptr.push_back((int64_t)sv.tgt.size());
  }
  fa.ptr.push_back((int64_t)fa.src.size());
  sv.ptr.push_back((int64_t)sv.src.size());
  // what a factorization clears
  std::vector<std::pair<int64_t, int64_t>> used;
  for (int64_t J = 0; J < sy.nsn; ++J)
    used.emplace_back(sy.front_off[J], rows(J) * (out.child[J] ? pivots(J) : rows(J)));
  std::sort(used.begin(), used.end());
  std::vector<int64_t> seg;
  for (size_t k = 0; k < used.size();) {
    const int64_t o = used[k].first;
    int64_t e = o;
    for (; k < used.size() && used[k].first <= e + 32; ++k) e = std::max(e, used[k].first + used[k].second);
    for (int64_t x = o; x < e; x += kSegment) {
      seg.push_back(x);
      seg.push_back(std::min(kSegment, e - x));
    }
  }
  out.nseg = (int64_t)seg.size() / 2;
  out.seg = ar.upload(seg.data(), (int64_t)seg.size());
  out.src = ar.upload(src.data(), (int64_t)src.size());
  out.map0 = ar.upload(map0.data(), (int64_t)map0.size());
  out.cnt = ar.upload(cnt.data(), (int64_t)cnt.size());
  out.dpos = ar.upload(dpos.data(), (int64_t)dpos.size());
  out.map = ar.upload(map.data(), (int64_t)map.size());
  out.slot = ar.upload(slot.data(), (int64_t)slot.size());
  out.front = ar.upload(front.data(), (int64_t)front.size());
  return out.seg && out.src && out.map0 && out.cnt && out.dpos && out.map && out.slot && out.front ? CLR_OK : CLR_E_OOM;
}

template <typename T>
void ThinSyrkOps<T>::clear_pool(cudaStream_t st, const ThinSyrk& ts, T* F) {
  k_clear_segments<T><<<(unsigned)ts.nseg, 256, 0, st>>>(F, ts.seg);
}

template <typename T>
void ThinSyrkOps<T>::add_level(cudaStream_t st, const ThinSyrk& ts, int64_t l, T* F, const T* Dp, T* W, T* part,
                               const int* skip) {
  for (const ThinSyrkParent& p : ts.lev[l]) {
    k_scatter_columns<T><<<(unsigned)((p.K * 32 + NT - 1) / NT), NT, 0, st>>>(F, W, p, ts.src, ts.map0, ts.cnt, ts.map,
                                                                              skip);
    k_syrk_tiles<T><<<dim3((unsigned)p.tiles, (unsigned)p.splits), NT, 0, st>>>(F, Dp, W, p, ts.dpos, part, skip);
    if (p.splits > 1)
      k_add_tiles<T><<<(unsigned)(p.tiles * (TB * TB / NT)), NT, 0, st>>>(F, p, part, skip);
  }
}

template <typename T>
void ThinSyrkOps<T>::fwd_level(cudaStream_t st, const ThinSyrk& ts, int64_t l, const T* F, const T* W, T* part, T* w,
                               const int64_t* sn_ptr, const int64_t* row_ptr, const int64_t* front_off,
                               const int64_t* upd_off, const int* skip) {
  for (const ThinSyrkParent& p : ts.lev[l]) {
    if (p.many)
      k_leaf_fwd<T><<<(unsigned)((p.nfront * 32 + NT - 1) / NT), NT, 0, st>>>(F, w, ts.front + p.front0, p.nfront, sn_ptr,
                                                                              row_ptr, front_off, upd_off, skip);
    k_panel_product<T><<<dim3((unsigned)((p.fP + NT - 1) / NT), (unsigned)p.vsplits), NT, 0, st>>>(W, w, p, ts.slot, part,
                                                                                                  skip);
    k_panel_add<T><<<(unsigned)((p.fP * 8 + NT - 1) / NT), NT, 0, st>>>(w, p, part, skip);
  }
}

template <typename T>
void ThinSyrkOps<T>::bwd_level(cudaStream_t st, const ThinSyrk& ts, int64_t l, const T* F, const T* Dp, const T* w, T* xs,
                               const int64_t* sn_ptr, const int64_t* row_ptr, const int64_t* front_off,
                               const int64_t* upd_off, const int32_t* rows_kkt, const int* skip) {
  for (const ThinSyrkParent& p : ts.lev[l])
    k_leaf_bwd<T><<<(unsigned)((p.nfront * 32 + NT - 1) / NT), NT, 0, st>>>(
        F, Dp, w, xs, ts.front + p.front0, p.nfront, sn_ptr, row_ptr, front_off, upd_off, rows_kkt, skip);
}

template struct ThinSyrkOps<float>;
template struct ThinSyrkOps<double>;
}  // namespace clr
