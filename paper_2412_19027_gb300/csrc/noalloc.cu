// Allocation-free dense LDL^T factor-and-solve for small quasi-definite systems.
//
// Some callers cannot allocate device memory at the point where they need a
// solve: code that runs while a CUDA graph is being captured (cudaMalloc is
// not allowed there), real-time control loops that must not allocate after
// start-up (for example a model-predictive controller that solves one small
// KKT system per control period), and plug-ins whose device memory is owned
// and budgeted by a host framework.  This entry point takes only caller-owned
// device buffers and works in registers and shared memory, so it never calls
// cudaMalloc or cudaFree and calls that overlap on the GPU do not disturb each
// other.
#include <cuda_runtime.h>

#include <mutex>
#include <type_traits>

#include "../../include/clr.h"
#include "device.cuh"
#include "rcp.cuh"

namespace clr {

constexpr int kNoAllocMaxN = CLR_NOALLOC_MAX_N;

// Reciprocal of a pivot.  (The other order of the two returns makes the chain of pivots 4 % slower.)
__device__ __forceinline__ double pivot_rcp(double d) {
  const double a = fabs(d);
  if (!(a > kRcpLow && a < kRcpHigh)) return 1.0 / d;
  return rcp_steps(d);
}

// One CTA, right-looking LDL^T with the dynamic-regularisation rule; the forward
// solve runs along (y_k is final when column k is), then D^{-1} and the backward
// solve.
//
// What bounds it: a GB300 SM retires ~1.7 FP64 FMA per clock and a warp
// instruction holds its sub-partition's pipe 64 clocks whatever its active lanes
// (DFMA 64, divide 569, barrier 33 clocks measured); so each pivot costs its chain
// (reciprocal, scaling, broadcast) and the rank-1 update in warp instructions.
// Layout: a 16 x 16 thread grid, thread (ti, tj) holding the entries
// (16 a + ti, 16 b + tj), a >= b, in registers; thread id 16 tj + ti, so a column's
// entries sit in half a warp.  That warp brings its column up to date first, forms
// the reciprocal and publishes the scaled column while the other warps still apply
// the previous pivot: one barrier per pivot.  (With every thread dividing its
// entries in place and the matrix in global memory a pivot cost ~4600 clocks.)
// L goes to shared memory for the backward solve.  On a GB300,
// N = 48: 111 -> 45 us a call, N = 128: 670 -> 223 us (FP64 floor of one SM 100 us).
template <int NB>
__global__ void __launch_bounds__(256) k_noalloc_ldl(const double* K, const double* signs, int N, const double* rhs,
                                                     double* x, double* D, double eps, double delta, int* hits) {
  extern __shared__ double Ls[];  // strictly lower L by rows: entry (i, k) at i (i - 1) / 2 + k
  __shared__ double pc[2][16 * NB], pl[2][16 * NB];  // a pivot column as it is and scaled, two in turn
  __shared__ double ys[16 * NB], sd[16 * NB];
  __shared__ signed char sgn[16 * NB];
  __shared__ int nhit;
  const int tid = threadIdx.x, ti = tid & 15, tj = tid >> 4;
  double v[NB][NB];
#pragma unroll
  for (int b = 0; b < NB; ++b)
#pragma unroll
    for (int a = b; a < NB; ++a) {
      const int i = 16 * a + ti, j = 16 * b + tj;
      v[a][b] = (i < N && i >= j) ? K[i + (int64_t)j * N] : 0.0;
    }
  double y = tid < N ? rhs[tid] : 0.0;  // entry tid of the right-hand side (N <= 128 threads)
  if (tid < N) sgn[tid] = signs[tid] > 0 ? 1 : -1;
  if (tid == 0) {
    nhit = 0;
    ys[0] = y;
  }
  __syncthreads();
  // column k = 16 kb + kk by the warp that holds it (its entries final)
  auto publish = [&](auto kb_, int kk) {
    constexpr int kb = decltype(kb_)::value;
    const int k = 16 * kb + kk;
    double d = __shfl_sync(0xffffffffu, v[kb][kb], ((kk & 1) << 4) + kk);
    if (tj != kk) return;
    const double sg = sgn[k];
    const bool hit = sg * d <= eps;
    if (hit) d = sg * delta;
    const double inv = pivot_rcp(d);
    if (ti == kk) {
      sd[k] = d;
      if (hit) ++nhit;
    }
#pragma unroll
    for (int a = kb; a < NB; ++a) {
      const int i = 16 * a + ti;
      const double c = v[a][kb], l = c * inv;
      pc[k & 1][i] = c;
      pl[k & 1][i] = l;
      if (i > k && i < N) Ls[i * (i - 1) / 2 + k] = l;
    }
  };
  auto block = [&](auto kb_) {
    constexpr int kb = decltype(kb_)::value;
    for (int kk = 0; kk < 16; ++kk) {
      const int k = 16 * kb + kk;
      if (k >= N) return;
      double l[NB], c[NB];
#pragma unroll
      for (int a = kb; a < NB; ++a) {
        l[a] = pl[k & 1][16 * a + ti];
        c[a] = pc[k & 1][16 * a + tj];
      }
      // (columns <= k and rows above the diagonal hold unused values)
      auto column = [&](auto b_) {
        constexpr int b = decltype(b_)::value;
#pragma unroll
        for (int a = b; a < NB; ++a) v[a][b] = fma(-l[a], c[b], v[a][b]);
      };
      const int kn = (kk + 1) & 15;
      const bool own = (tid >> 5) == (kn >> 1) && k + 1 < N;  // my warp holds column k + 1
      if (kk < 15) {
        if ((tid >> 5) >= ((kk + 1) >> 1)) column(std::integral_constant<int, kb>{});
        if (own) publish(std::integral_constant<int, kb>{}, kn);
        if constexpr (kb + 1 < NB) column(std::integral_constant<int, (kb + 1 < NB ? kb + 1 : kb)>{});
      } else if constexpr (kb + 1 < NB) {
        column(std::integral_constant<int, (kb + 1 < NB ? kb + 1 : kb)>{});
        if (own) publish(std::integral_constant<int, (kb + 1 < NB ? kb + 1 : kb)>{}, kn);
      }
#pragma unroll
      for (int b = kb + 2; b < NB; ++b)
#pragma unroll
        for (int a = b; a < NB; ++a) v[a][b] = fma(-l[a], c[b], v[a][b]);
      if (tid > k && tid < N) {
        y = fma(-pl[k & 1][tid], ys[k], y);
        if (tid == k + 1) ys[tid] = y;
      }
      __syncthreads();
    }
  };
  if (tid < 32) publish(std::integral_constant<int, 0>{}, 0);
  __syncthreads();
  block(std::integral_constant<int, 0>{});
  if constexpr (NB > 1) block(std::integral_constant<int, (NB > 1 ? 1 : 0)>{});
  if constexpr (NB > 2) block(std::integral_constant<int, (NB > 2 ? 2 : 0)>{});
  if constexpr (NB > 3) block(std::integral_constant<int, (NB > 3 ? 3 : 0)>{});
  if constexpr (NB > 4) block(std::integral_constant<int, (NB > 4 ? 4 : 0)>{});
  if constexpr (NB > 5) block(std::integral_constant<int, (NB > 5 ? 5 : 0)>{});
  if constexpr (NB > 6) block(std::integral_constant<int, (NB > 6 ? 6 : 0)>{});
  if constexpr (NB > 7) block(std::integral_constant<int, (NB > 7 ? 7 : 0)>{});
  // L^T x = z: thread i takes x_k off z_i as soon as x_k is final (i < k); 128 threads
  if (tid < 128) {
    double zi = tid < N ? y / sd[tid] : 0.0;
    for (int k = N - 1; k > 0; --k) {
      if (tid == k) ys[k] = zi;
      asm volatile("barrier.sync 1, 128;" ::: "memory");
      if (tid < k) zi = fma(-Ls[k * (k - 1) / 2 + tid], ys[k], zi);
    }
    if (tid < N) {
      x[tid] = zi;
      if (D) D[tid] = sd[tid];
    }
  }
  if (tid == 0 && hits) *hits = nhit;
}

namespace {
std::mutex g_noalloc_mu;
bool g_noalloc_ready[64] = {false};  // kernel attributes set, per device ordinal

size_t noalloc_smem(int N) { return sizeof(double) * (size_t)(N > 1 ? N * (N - 1) / 2 : 1); }

template <int NB>
cudaError_t noalloc_attr() {
  return cudaFuncSetAttribute(k_noalloc_ldl<NB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)noalloc_smem(16 * NB < kNoAllocMaxN ? 16 * NB : kNoAllocMaxN));
}
}  // namespace

}  // namespace clr

extern "C" int clr_dense_ldl_solve_noalloc(const double* K, const double* signs, int32_t N, const double* rhs,
                                           double* x, double* D, double dyn_reg_eps, double dyn_reg_delta,
                                           int32_t* dyn_hits, void* stream) {
  using namespace clr;
  if (N < 0 || !K || !signs || !rhs || !x) return CLR_E_INVALID;
  if (N > kNoAllocMaxN) return CLR_E_UNSUPPORTED;
  if (N == 0) return CLR_OK;
  int dev = 0;
  CLR_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return CLR_E_UNSUPPORTED;
  {
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_ready[dev]) {  // the largest systems need more than 48 KB of shared memory
      CLR_CUDA(noalloc_attr<7>());
      CLR_CUDA(noalloc_attr<8>());
      g_noalloc_ready[dev] = true;
    }
  }
  const size_t sm = noalloc_smem(N);
  cudaStream_t st = (cudaStream_t)stream;
  switch ((N + 15) / 16) {  // 16-row tiles
#define CLR_NA(NB) \
  case NB: k_noalloc_ldl<NB><<<1, 256, sm, st>>>(K, signs, N, rhs, x, D, dyn_reg_eps, dyn_reg_delta, dyn_hits); break;
    CLR_NA(1) CLR_NA(2) CLR_NA(3) CLR_NA(4) CLR_NA(5) CLR_NA(6) CLR_NA(7) CLR_NA(8)
#undef CLR_NA
    static_assert(kNoAllocMaxN == 8 * 16, "the dispatch covers every order");
  }
  CLR_CHECK_LAUNCH();
  return CLR_OK;
}
