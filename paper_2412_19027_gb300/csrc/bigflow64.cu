// Dataflow factorization of the large FP64 fronts of one level with their 64 x 64 x 64
// products on the tensor cores.
//
// What bounds the FMA version (bigflow.cu): a GB300 SM retires ~1.7 FP64 FMA per clock, so a
// 64^3 product is 75 us of one SM's FP64 pipe; the FP64 tensor instruction runs no faster
// (684 clocks per 8 x 8 x 4).  Here each FP64 operand is cut into seven 8-bit digits that
// tcgen05 kind::f16 multiplies exactly, and the sums are put together again in integers
// (the error-free splitting of Ozaki, Ogita, Oishi and Rump, "Error-free transformations of
// matrix multiplication by using fast routines of matrix multiplication and its
// applications", Numer. Algorithms 59, 2012):
//   - row r of an operand is scaled by a power of two so that its largest entry is below
//     2^55 as an integer, X = rint(x 2^(55 - e_r)), and written in balanced base 256,
//     X = sum_s d_s 256^(6 - s), |d_s| <= 128 (exact in FP16);
//   - the products of digit matrices s and t of equal s + t <= 7 are summed in one FP32
//     accumulator in tensor memory: at most 4 products of 64 terms up to 2^14, so every
//     partial sum is an integer up to 2^22, exact in FP32;
//   - the eight sums G_0 .. G_7 give (X Y) / 2^54 as a 64-bit integer, which is normalised to a
//     double in integer arithmetic; one FP64 addition per entry remains.  Left out are the digit
//     products with s + t >= 8: five of s + t = 8, at most 2^-55.7 of the product of the row maxima
//     over 64 terms.
// Before splitting, the shared index k is scaled by a power of two on one side and its inverse
// on the other, so that both operands are rows of sqrt(D)-scaled factors:
//   - U and EU: rows of L |D|^(1/2).  The rounding of a product is 2^-55 of (the largest entry of
//     row i) times (the sum over row j), and the same with i and j exchanged: the size of
//     n u |L| |D| |L|^T, the error of any LDL^T, for rows whose large entries meet in the same columns.
//   - T, Efin and the block's own inverse, products with V = L_KK^{-1}: column l of V is scaled by
//     sqrt(F_ll).  In a block of one sign |F_il| <= sqrt(F_ii F_ll), as in a Cholesky factorization, and
//     |d_l| <= |F_ll|.  In a block of both signs a pivot can grow from a tiny diagonal (the
//     regularisation of an equality row or of an LP variable), and its column would set every row's
//     maximum; so where a pivot has grown the columns are raised as far as no row of V 2^g gets a larger
//     maximum than e_k = max(sqrt|d_k|, max_l |V_kl| sqrt(F_ll)).
// Against FMA products (NumPy emulation, n = 192, 32 systems each, geometric means): the error of the
// factorization, 0.5 to 0.94 times theirs on all of the following; the residual of one unrefined solve,
// in brackets with sqrt(F_ll) alone: both signs in every block, equality rows regularised by 1e-8 1.0 (36),
// LP with a scaling over 4 decades 0.7 (0.75), more rows than variables 0.8 (2.1); definite with a
// spectrum over 14 decades 0.55; but 3.2 (45) for LP with a scaling over 12 decades and 7.8 for the
// block of a PSD cone at the end of a solve (scaling over 12 decades): there U's rounding relative to the
// row's maximum counts (4.0 and 3.7 by itself), where FMAs keep the 53 bits of each entry.  Refinement
// removes it; schedule 2 has FMA products.  A row with an entry that is not finite gives NaN in its
// results.
//
// Tasks and waits are those of bigflow.cu without the fused or split chain task: D(p), T(p, i),
// Efin(p, e), U(p, i, j), EU(p, i, e).  Producers store their tile also as digits ("packs",
// 56 KB in the MMA's layout, copied to shared memory by cp.async.bulk):
//   PA(p, i) = L_IK 2^h, PB(p, i) = (L_IK D_K) 2^-h (h_k = half the exponent of d_k),
//   PE(p, e) = E_KC^T 2^-h, PT(p) = Linv 2^g (g_l = half the exponent of F_ll, raised where pivots grew), so that
//   U: F_IJ -= PA(p, i) PB(p, j)^T;  EU: E_IC -= PA(p, i) PE(p, e)^T;
//   T: L_IK = (F_IK 2^-g) PT(p)^T D^{-1};  Efin: E_KC^T <- (E_KC^T 2^-g) PT(p)^T,
// with F_IK and E_KC^T split in the task.  One CTA per SM (512 columns of tensor memory).
// Per task on a GB300 (front of 2052 rows; FMA version in brackets): D 64 us (95), T 24 (41), Efin 18
// (57), U 11 (57), EU 11 (57); the front: 3.7 ms.
#include <algorithm>

#include "bfdiag.cuh"
#include "bigfront.cuh"
#include "flowsync.cuh"

namespace clr {
namespace {
constexpr int NB = kBfNB;
constexpr int NT = kFlowThreads;
constexpr int kSlice = NB * NB * 2;                   // one digit matrix, FP16: 8 KB
constexpr int kDig = 7;
constexpr int kPackBytes = kDig * kSlice;             // 57344
constexpr int kTileStride = (int)kPack64Bytes;        // digits, then 64 row exponents, g[64], h[64]
static_assert(kTileStride == kPackBytes + 3 * 64 * 4 && kTileStride % 16 == 0, "pack layout");
constexpr int kBad = 1 << 20;                         // row exponent of a row with a value that is not finite
// shared memory: A digits (an eighth matrix of zeros pairs with the seventh), B digits, scratch
constexpr int kOffB = 8 * kSlice, kOffS = kOffB + kPackBytes;
// scratch: D(p)'s blocks, or two 64 x 64 tiles of doubles: entry (row, k) at tile_at(k) + row
constexpr int kTile = 64 * 65 + 3 * 8;
__device__ __forceinline__ int tile_at(int k) { return k * 65 + (k >> 4) * 8; }
constexpr int kScratch = 2 * kTile * 8;
static_assert(2 * kTile >= kDiagSmem, "scratch");
constexpr size_t kSmem = (size_t)kOffS + kScratch + 1024;

__device__ __forceinline__ uint32_t s_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void fence_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }
__device__ __forceinline__ void fence_async_shared() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// K-major core matrices of 8 rows x 16 bytes, adjacent in K 128 bytes apart and in rows 1024
__device__ __forceinline__ uint64_t dig_desc(uint32_t a) {
  uint64_t d = (uint64_t)((a & 0x3FFFF) >> 4);
  d |= (uint64_t)(128 >> 4) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;  // tcgen05 descriptor version; no swizzle, base offset 0
  return d;
}
// M = 128, N = 64, D FP32, A and B FP16, both K-major
constexpr uint32_t kF16Idesc = (1u << 4) | ((uint32_t)(64 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
__device__ __forceinline__ void mma_f16(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(ad), "l"(bd), "r"(kF16Idesc), "r"(acc));
}
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

// exponent of |x| as in |x| < 2^(ilog + 1) (zero and subnormals: very small; not finite: kBad)
__device__ __forceinline__ int ilog_of(double x) {
  const int e = (__double2hiint(x) >> 20) & 0x7ff;
  return e == 0 ? -kBad : (e == 0x7ff ? kBad : e - 1023);
}
// rint(x 2^(sh + 55 - e)) plus 128 in each of seven bytes, for |x| 2^sh < 2^e
__device__ __forceinline__ uint64_t digits_of(double x, int sh, int e) {
  constexpr uint64_t bias = 0x0080808080808080ull;
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  if (ex == 0 || ex == 0x7ff) return bias;
  const uint64_t m = (b & 0xfffffffffffffull) | 0x10000000000000ull;
  const int s = e - 3 - (ex - 1023 + sh);  // X = m 2^-s, s >= -2
  uint64_t X;
  if (s <= 0) X = m << (-s & 3);
  else X = s > 54 ? 0ull : (m + (1ull << (s - 1))) >> s;
  return (int64_t)b < 0 ? bias - X : bias + X;
}

// All threads: the 64 x 64 matrix with entry (r, k) at Y[r rs + k ks + (k >> 4) sk], its
// k-th column scaled by 2^(sgn sh[k]), as digits at dst + s kSlice + ... (global or shared) and
// row exponents at `exps`.  Ends without a barrier.  One copy of the code, in loops: with everything
// unrolled and inlined the kernel's code was 430 KB and its tasks waited for instructions
// (a CTA's first task of a kind took twice the time of the later ones).
__device__ __noinline__ void pack_tile(const double* Y, int rs, int ks, int sk, const int* sh, int sgn,
                                       unsigned char* dst, int* exps) {
  const int lane = threadIdx.x & 31, r = 8 * (threadIdx.x >> 5) + (lane & 7), kq = lane >> 3;
  const double* y = Y + r * rs + 16 * kq * ks + kq * sk;
  const int* shk = sh + 16 * kq;
  int m = -kBad;
#pragma unroll 4
  for (int u = 0; u < 16; ++u) {
    const int l = ilog_of(y[u * ks]);
    m = max(m, l >= kBad ? kBad : (l <= -kBad ? -kBad : l + sgn * shk[u]));
  }
  m = max(m, __shfl_xor_sync(~0u, m, 8));
  m = max(m, __shfl_xor_sync(~0u, m, 16));
  const int e = m >= kBad ? kBad : (m <= -kBad ? 0 : m + 1);
  if (kq == 0) exps[r] = e;
#pragma unroll 1
  for (int g = 0; g < 2; ++g) {
    uint64_t z[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) z[u] = digits_of(y[(8 * g + u) * ks], sgn * shk[8 * g + u], e);
    unsigned char* d = dst + (r >> 3) * 1024 + (2 * kq + g) * 128 + (r & 7) * 16;
#pragma unroll
    for (int s = 0; s < kDig; ++s) {
      const int q = 6 - s;  // byte of the digit
      uint32_t o[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const uint32_t wa = q < 4 ? (uint32_t)z[2 * v] : (uint32_t)(z[2 * v] >> 32);
        const uint32_t wb = q < 4 ? (uint32_t)z[2 * v + 1] : (uint32_t)(z[2 * v + 1] >> 32);
        // FP16 1024 + byte, then minus 1152: the digit
        // (the first digit is up to 128: nine bits)
        const uint32_t t = __byte_perm(wa, wb, (q & 3) | ((4 + (q & 3)) << 4));
        const uint32_t h = s == 0 ? __byte_perm(wa, wb, 0x7632) | 0x64006400u : __byte_perm(t, 0x64646464u, 0x4140);
        asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(o[v]) : "r"(h), "r"(0x64806480u));
      }
      *reinterpret_cast<uint4*>(d + s * kSlice) = make_uint4(o[0], o[1], o[2], o[3]);
    }
  }
}

// Thread 0: the 19 digit products of A (at sA) and B (at sB) into tensor memory.  A MMA takes
// two neighbouring digits of A as 128 rows: block t (64 columns) gets the products of digit sum t
// in lanes 0-63 and those of digit sum t + 1 with the odd digits of A in lanes 64-127.
__device__ __forceinline__ void issue_products(uint32_t sA, uint32_t sB, uint32_t tmem, uint32_t bar) {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
  for (int t = 0; t < 8; ++t) {
    uint32_t acc = 0;
#pragma unroll 1
    for (int i = 0; i < 8; i += 2) {
      const int j = t - i;
      if (j < 0 || j >= kDig) continue;
#pragma unroll
      for (int ks = 0; ks < NB / 16; ++ks) {
        mma_f16(tmem + 64u * t, dig_desc(sA + i * kSlice + 256u * ks), dig_desc(sB + j * kSlice + 256u * ks), acc);
        acc = 1;
      }
    }
  }
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// v 2^e as a double, rounded to nearest, ties to even (zero below the normal range)
__device__ __forceinline__ double scaled_double(long long v, int e) {
  const uint64_t mag = v < 0 ? (uint64_t)-v : (uint64_t)v;
  const int lz = __clzll((long long)mag);
  const uint64_t n = mag << (lz & 63);
  uint64_t m = n >> 11;
  const uint64_t rest = n & 0x7ff;
  m += (rest > 0x400 || (rest == 0x400 && (m & 1))) ? 1 : 0;
  const int ex = 63 - lz + e + 1023;                 // exponent field of the leading bit
  uint64_t bits = ((uint64_t)(ex - 1) << 52) + m;    // (a carry out of m raises the exponent)
  if (mag == 0 || ex < 1) bits = 0;
  if (ex > 2046) bits = 0x7ff0000000000000ull;
  if (e > kBad / 2) bits = 0x7ff8000000000000ull;
  if (v < 0) bits |= 0x8000000000000000ull;
  return __longlong_as_double((long long)bits);
}

// the integer of an FP32 accumulator with |v| <= 2^22
__device__ __forceinline__ int acc_int(uint32_t b) {
  return __float_as_int(__uint_as_float(b) + 12582912.0f) - 0x4B400000;
}

// eight columns of four neighbouring 64-column blocks
__device__ __forceinline__ void tmem_ld8x4(uint32_t a, uint32_t (&v)[4][8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%32];\n"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%33];\n"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%16,%17,%18,%19,%20,%21,%22,%23}, [%34];\n"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%24,%25,%26,%27,%28,%29,%30,%31}, [%35];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(v[0][0]), "=r"(v[0][1]), "=r"(v[0][2]), "=r"(v[0][3]), "=r"(v[0][4]), "=r"(v[0][5]), "=r"(v[0][6]), "=r"(v[0][7]), 
        "=r"(v[1][0]), "=r"(v[1][1]), "=r"(v[1][2]), "=r"(v[1][3]), "=r"(v[1][4]), "=r"(v[1][5]), "=r"(v[1][6]), "=r"(v[1][7]), 
        "=r"(v[2][0]), "=r"(v[2][1]), "=r"(v[2][2]), "=r"(v[2][3]), "=r"(v[2][4]), "=r"(v[2][5]), "=r"(v[2][6]), "=r"(v[2][7]), 
        "=r"(v[3][0]), "=r"(v[3][1]), "=r"(v[3][2]), "=r"(v[3][3]), "=r"(v[3][4]), "=r"(v[3][5]), "=r"(v[3][6]), "=r"(v[3][7])
      : "r"(a), "r"(a + 64), "r"(a + 128), "r"(a + 192)
      : "memory");
}

// All threads, after the MMAs: the product as doubles in the tile X (eA, eB: row exponents of the
// operands; entry (r, c) at tile_at(c) + r); X2: a second tile.  Ends with a barrier.
__device__ __forceinline__ void read_products(uint32_t tmem, const int* eA, const int* eB, double* X, double* X2) {
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31, q = wid & 3, h = wid >> 2;
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const bool top = q < 2;  // lanes 0-63: digit sum t; 64-127: t + 1
  const uint32_t base = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(32 * h);
  const int r = 32 * (q & 1) + lane;
  long long* P = reinterpret_cast<long long*>(top ? X : X2) + r;
#pragma unroll 1
  for (int g = 0; g < 4; ++g) {
    // units of 2^-54 X Y: digit sum s has weight 2^(42 - 8 s)
    uint32_t a[4][8], b[4][8];
    tmem_ld8x4(base + 8 * g, a);        // digit sums 0 .. 3 (top) or 1 .. 4
    tmem_ld8x4(base + 256 + 8 * g, b);  // 4 .. 7 or 5 .. 7 (the last block's lower half is not read)
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      long long T = 0;
#pragma unroll
      for (int t = 0; t < 4; ++t) T = T * 256 + acc_int(a[t][c]);
      T = T * 256 + acc_int(b[0][c]);
      const int i5 = acc_int(b[1][c]), i6 = __float2int_rn(__uint_as_float(b[2][c]));
      const int lo = top ? i6 * 256 + acc_int(b[3][c]) : i5 * 256 + i6;
      T = (top ? T * 1024 + (long long)i5 * 4 : T * 4) + ((lo + 8192) >> 14);
      P[tile_at(32 * h + 8 * g + c)] = T;
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  const int c0 = 32 * h + (top ? 0 : 16), er = eA[r];
#pragma unroll 4
  for (int u = 0; u < 16; ++u) {
    const int at = tile_at(c0 + u) + r;
    const long long v = __double_as_longlong(X[at]) + __double_as_longlong(X2[at]);
    X[at] = scaled_double(v, er + eB[c0 + u] - 56);
  }
  __syncthreads();
}

// 27-bit low and 28-bit high parts x0, x1 of the integer rint(x 2^(sh + 55 - e)), |x| 2^sh < 2^e
__device__ __forceinline__ int2 halves_of(double x, int sh, int e) {
  constexpr int64_t bias = 0x0080808080808080ll;
  const int64_t X = (int64_t)digits_of(x, sh, e) - bias;
  const int x1 = (int)((X + (1ll << 26)) >> 27);
  return make_int2((int)(X - ((int64_t)x1 << 27)), x1);
}
// Exact dot product of 16 terms of such rows in 64-bit integers: four IMAD.WIDE a term (an FP64
// FMA takes 64 clocks of its pipe per warp); the sum is value() 2^(e_a + e_b - 56).
struct IntDot {
  long long hh = 0, mid = 0, ll = 0;
  __device__ __forceinline__ void add(int2 a, int2 b) {
    hh += (long long)a.y * b.y;
    mid += (long long)a.y * b.x;
    mid += (long long)a.x * b.y;
    ll += (long long)a.x * b.x;
  }
  __device__ __forceinline__ long long value() const { return hh + ((mid + (ll >> 27) + (1ll << 26)) >> 27); }
};

// integers in the order of the doubles (NaN above all): no FP64 compare
__device__ __forceinline__ long long order_key(double x) {
  const long long b = __double_as_longlong(x);
  const bool nan = (b & 0x7fffffffffffffffll) > 0x7ff0000000000000ll;
  return nan ? 0x7fffffffffffffffll : (b < 0 ? b ^ 0x7fffffffffffffffll : b);
}
// 1 / d to about half an ulp in integers (~110 clocks; two FP64 steps on the estimate: 230): with
// m in [1, 2) the mantissa of d and y0 the hardware's estimate of 1 / m (20 bits), e = 1 - m y0
// is exact in 64 bits and 1 / m = y0 (1 + e + e^2) to 2^-57.
__device__ __forceinline__ double rcp_pivot(double d) {
  const long long b = __double_as_longlong(d);
  const int ex = (int)((b >> 52) & 0x7ff);
  if (ex < 2 || ex > 2043) return 1.0 / d;
  const unsigned long long M = ((unsigned long long)b & 0xfffffffffffffull) | 0x10000000000000ull;
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;"
      : "=d"(y)
      : "d"(__longlong_as_double((long long)((M & 0xfffffffffffffull) | 0x3ff0000000000000ull))));
  const unsigned long long yb = (unsigned long long)__double_as_longlong(y);
  // y in [1/2, 1]: Y0 = y 2^21, cut to an integer
  const int ye = (int)(yb >> 52);  // 1022 or 1023
  const unsigned Y0 = (unsigned)(((yb & 0xfffffffffffffull) | 0x10000000000000ull) >> (52 - 21 + 1023 - ye));
  const long long e73 = -(long long)(M * Y0);                // e 2^73 (2^73 = 0 modulo 2^64)
  const int e40 = (int)(e73 >> 33);
  const long long c58 = (e73 >> 15) + (((long long)e40 * e40) >> 22);  // (e + e^2) 2^58
  const long long Y = ((long long)Y0 << 41) + ((c58 * (long long)Y0) >> 17);  // y 2^62
  const unsigned long long m = (unsigned long long)((Y + 256) >> 9);
  // 1/d = (m / 2^53) 2^(1023 - ex): m carries the hidden bit
  const unsigned long long r = ((unsigned long long)(2044 - ex) << 52) + m;
  return __longlong_as_double((long long)(r | ((unsigned long long)b & 0x8000000000000000ull)));
}

constexpr int kLI = 65;  // row strides of the integer operands (int2; odd: no bank conflicts)
constexpr int kLP = 17;
struct Diag64Smem {
  int2 ia[64 * kLI];       // L 2^h by rows, exponents ea[panel][row]
  int2 iq[16 * kLP];       // Linv_QQ 2^g by rows, exponents eq
  int2 ix[48 * kLP];       // X 2^-g by columns, exponents ex
  double cb[8 * 64];       // pivot columns: four of this group of columns, four of the last
  int ea[4 * 64], eq[16], ex[48], xm[2 * 64], gq[4 * 16];
};
struct Diag64SmemB {
  int2 ib[2 * 64 * kLP];   // (L d) 2^-h of a panel by rows, exponents eb[row], for two panels
  int2 ic[48 * kLI];       // L^{-1} 2^-h by columns, exponents ec[block row][column]
  int eb[2 * 64], ec[3 * 48];
  double x[16 * 49];       // X = sum_M L_QM Linv_M
};
static_assert(sizeof(Diag64Smem) <= kPackBytes && sizeof(Diag64SmemB) <= kPackBytes, "scratch");
__device__ __forceinline__ int row_exp(int m) { return m >= kBad ? kBad : (m <= -kBad ? 0 : m + 1); }
// the scale of a column whose largest entry has exponent m
__device__ __forceinline__ int block_scale(int m) { return m <= -kBad || m >= kBad ? 0 : -m; }
__device__ __forceinline__ int shifted(double x, int sh) {
  const int l = ilog_of(x);
  return l >= kBad ? kBad : (l <= -kBad ? -kBad : l + sh);
}

// Pivots 16 q .. 16 q + 15 by four warps (barrier 2): NP = 2: rows 32 (wid & 1) + lane, columns of
// parity wid >> 1; NP = 4 (q >= 2: rows 0-31 are done): rows 32 + lane, columns wid modulo 4.
// Groups of four columns: a pivot updates its group at once, the columns after it by the group's
// four pivots together (an FMA behind its own load and branch took 150 clocks, in a batch 85).
template <int NP>
__device__ __forceinline__ void diag64_panel(int q, int pw, double* A, Diag64Smem& sa, Diag64SmemB& sb,
                                             DiagScratch<double>& sh, int* hs, long long key_eps, double delta,
                                             double rdelta, int& nhit) {
  constexpr int LD = kDiagLD, NC = 16 / NP, GC = 4 / NP;
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31, c0 = 16 * q;
  const int row = NP == 2 ? 32 * (wid & 1) + lane : 32 + lane, par = NP == 2 ? wid >> 1 : wid;
  constexpr long long kSign = (long long)0x8000000000000000ull;
  double v[NC], dk = 0.0;
  int2* ib = sb.ib + (q & 1) * 64 * kLP;
  double* cd = reinterpret_cast<double*>(ib);  // this thread's entries of L d, then their integers in place
#pragma unroll
  for (int t = 0; t < NC; ++t) v[t] = A[row * LD + c0 + NP * t + par];
  if (par == 0) sa.xm[row] = sa.xm[64 + row] = -kBad;
#pragma unroll 1
  for (int g = 0; g < 4; ++g) {
    double* cg = sa.cb + 256 * (g & 1);
    double ml[4];
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      const int k = 4 * g + o, kk = c0 + k;
      double* cc = cg + 64 * o;
      if (par == o % NP) cc[row] = v[o / NP];
      const bool ng = sh.sgn[kk] < 0;
      asm volatile("barrier.sync 2, 128;" ::: "memory");
      double d = cc[kk];
      const double cr = cc[row];
      // (the reciprocal does not wait for the test)
      double rd = rcp_pivot(d);
      const bool hit = kk < pw && order_key(__longlong_as_double(__double_as_longlong(d) ^ (ng ? kSign : 0ll))) <= key_eps;
      if (hit) d = ng ? -delta : delta, rd = ng ? -rdelta : rdelta;
      const double lr = cr * rd;
      ml[o] = __longlong_as_double(__double_as_longlong(lr) ^ kSign);
#pragma unroll
      for (int t = 0; t < GC; ++t)
        if (NP * t + NP - 1 > o && NP * t + par > o) v[t] = fma(ml[o], cc[c0 + 4 * g + NP * t + par], v[t]);
      if (par == o % NP) {
        if (row >= kk) A[row * LD + kk] = row == kk ? d : lr;
        cd[row * kLP + k] = cr;
      }
      if (lane == k) dk = d;
      nhit += hit ? 1 : 0;
    }
#pragma unroll
    for (int u = 1; u < 4; ++u) {
      if (g + u < 4) {
        const double* cp = cg + c0 + 4 * (g + u) + par;
        double w[4 * GC];
#pragma unroll
        for (int e = 0; e < 4 * GC; ++e) w[e] = cp[64 * (e / GC) + NP * (e % GC)];
#pragma unroll
        for (int e = 0; e < 4 * GC; ++e) v[GC * u + e % GC] = fma(ml[e / GC], w[e], v[GC * u + e % GC]);
      }
    }
#pragma unroll
    for (int t = 0; t + GC < NC; ++t) v[t] = v[t + GC];
  }
  if (wid == 0 && lane < 16) {
    sh.dv[c0 + lane] = dk;
    const int lg = ilog_of(dk);
    hs[c0 + lane] = lg <= -kBad || lg >= kBad ? 0 : lg >> 1;
  }
  // the integer operands L 2^h, (L d) 2^-h of the rows below
  // (their largest exponents here, not in the loop: integer work there is on the chain of pivots)
  asm volatile("barrier.sync 2, 128;" ::: "memory");
  int ma = -kBad, mb = -kBad;
#pragma unroll
  for (int t = 0; t < NC; ++t) {
    const int c = NP * t + par, h = hs[c0 + c];
    const int xl = shifted(A[row * LD + c0 + c], h), xd = shifted(cd[row * kLP + c], -h);
    if (row > c0 + c) ma = max(ma, xl), mb = max(mb, xd);
  }
  atomicMax(&sa.xm[row], ma);
  atomicMax(&sa.xm[64 + row], mb);
  asm volatile("barrier.sync 2, 128;" ::: "memory");
  const int xa = row_exp(sa.xm[row]), xb = row_exp(sa.xm[64 + row]);
  if (par == 0) {
    sa.ea[64 * q + row] = xa;
    sb.eb[64 * (q & 1) + row] = xb;
  }
#pragma unroll 2
  for (int t = 0; t < NC; ++t) {
    const int c = NP * t + par;
    const bool in = row > c0 + c;
    const double lv = in ? A[row * LD + c0 + c] : 0.0, cv = in ? cd[row * kLP + c] : 0.0;
    sa.ia[row * kLI + c0 + c] = halves_of(lv, hs[c0 + c], xa);
    ib[row * kLP + c] = halves_of(cv, -hs[c0 + c], xb);
  }
}

// 16 x 16 block (I, J) of the trailing matrix: a_rs -= sum_m l_rm (l_sm d_m) over panel q; 256 entries
__device__ __noinline__ void diag64_update(int q, int I, int J, int idx, double* A, const Diag64Smem& sa,
                                              const Diag64SmemB& sb) {
  const int r = 16 * I + (idx >> 4), s = 16 * J + (idx & 15);
  const int2* ib = sb.ib + (q & 1) * 64 * kLP;
  IntDot acc;
#pragma unroll 4
  for (int m = 0; m < 16; ++m) acc.add(sa.ia[r * kLI + 16 * q + m], ib[s * kLP + m]);
  if (r >= s)
    A[r * kDiagLD + s] -= scaled_double(acc.value(), sa.ea[64 * q + r] + sb.eb[64 * (q & 1) + s] - 56);
}

// Block row Q of L^{-1}, by the 128 threads of warps 4-7 (tid 0 .. 127 here, barrier 3): the inverse of
// L_QQ, Linv_QP = -Linv_QQ X_P, its operands (Q < 3), and X of block row Q + 1.
__device__ __noinline__ void diag64_inverse_row(int Q, int tid, const double* A, double* V, Diag64Smem& sa,
                                                   Diag64SmemB& sb, const int* gs, const int* hs) {
  constexpr int LD = kDiagLD;
  const int R0 = 16 * Q;
  auto bar = [] { asm volatile("barrier.sync 3, 128;" ::: "memory"); };
  {
    // both 8 x 8 diagonal blocks by column sweeps, lane: row 4 r + c of four columns; then the 8 x 8
    // block below them, -C^{-1} B A^{-1}
    const int w = tid >> 5, lane = tid & 31, o = R0 + 8 * (w >> 1), r = lane >> 2, c = 4 * (w & 1) + (lane & 3);
    double x = r == c ? 1.0 : 0.0;
#pragma unroll
    for (int m = 0; m < 7; ++m) {
      const double xm = __shfl_sync(~0u, x, 4 * m + (lane & 3));
      if (r > m) x = fma(-A[(o + r) * LD + o + m], xm, x);
    }
    V[(o + r) * LD + o + c] = x;
  }
  bar();
  if (tid < 64) {  // B A^{-1}
    const int r = R0 + 8 + (tid >> 3), c = R0 + (tid & 7);
    double s = 0.0;
#pragma unroll
    for (int m = 0; m < 8; ++m) s = fma(A[r * LD + R0 + m], V[(R0 + m) * LD + c], s);
    V[r * LD + c] = s;
  }
  bar();
  double b1 = 0.0;
  if (tid < 64) {
    const int r = R0 + 8 + (tid >> 3), c = R0 + (tid & 7);
#pragma unroll
    for (int m = 0; m < 8; ++m) b1 = fma(-V[r * LD + R0 + 8 + m], V[(R0 + 8 + m) * LD + c], b1);
  }
  bar();
  if (tid < 64) V[(R0 + 8 + (tid >> 3)) * LD + R0 + (tid & 7)] = b1;
  if (Q > 0) {
    bar();
    // rows of Linv_QQ (8 threads a row), columns of X (2 threads a column)
    const int a0 = tid >> 3, c0 = 2 * (tid & 7);
    const double x0 = V[(R0 + a0) * LD + R0 + c0], x1 = V[(R0 + a0) * LD + R0 + c0 + 1];
    const bool grown = __any_sync(~0u, hs[R0 + (tid & 15)] > gs[R0 + (tid & 15)]);
    if (grown) {  // as at the end of diag64, for this block
      int e = max(shifted(x0, gs[R0 + c0]), shifted(x1, gs[R0 + c0 + 1]));
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) e = max(e, __shfl_xor_sync(~0u, e, o));
      e = max(e, hs[R0 + a0]);
      int m0 = shifted(x0, -e), m1 = shifted(x1, -e);
#pragma unroll
      for (int o = 8; o < 32; o <<= 1) {
        m0 = max(m0, __shfl_xor_sync(~0u, m0, o));
        m1 = max(m1, __shfl_xor_sync(~0u, m1, o));
      }
      if ((tid & 31) < 8) {
        sa.gq[16 * (tid >> 5) + c0] = m0;
        sa.gq[16 * (tid >> 5) + c0 + 1] = m1;
      }
      bar();
    }
    auto g_of = [&](int k) {
      if (!grown) return gs[R0 + k];
      return block_scale(max(max(sa.gq[k], sa.gq[16 + k]), max(sa.gq[32 + k], sa.gq[48 + k])));
    };
    {
      const int g0 = g_of(c0), g1 = g_of(c0 + 1);
      int m = max(shifted(x0, g0), shifted(x1, g1));
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) m = max(m, __shfl_xor_sync(~0u, m, o));
      const int e = row_exp(m);
      if (c0 == 0) sa.eq[a0] = e;
      sa.iq[a0 * kLP + c0] = halves_of(x0, g0, e);
      sa.iq[a0 * kLP + c0 + 1] = halves_of(x1, g1, e);
    }
    if (tid < 2 * R0) {
      const int b = tid >> 1, k0 = 8 * (tid & 1);
      int m = -kBad;
#pragma unroll
      for (int k = 0; k < 8; ++k) m = max(m, shifted(sb.x[(k0 + k) * 49 + b], -g_of(k0 + k)));
      m = max(m, __shfl_xor_sync(~0u, m, 1));
      const int e = row_exp(m);
      if (k0 == 0) sa.ex[b] = e;
#pragma unroll
      for (int k = 0; k < 8; ++k) sa.ix[b * kLP + k0 + k] = halves_of(sb.x[(k0 + k) * 49 + b], -g_of(k0 + k), e);
    }
    bar();
    for (int idx = tid; idx < 16 * R0; idx += 128) {
      const int a = idx & 15, b = idx >> 4;
      IntDot acc;
#pragma unroll 4
      for (int m = 0; m < 16; ++m) acc.add(sa.iq[a * kLP + m], sa.ix[b * kLP + m]);
      V[(R0 + a) * LD + b] = -scaled_double(acc.value(), sa.eq[a] + sa.ex[b] - 56);
    }
  }
  bar();
  if (Q == 3) return;
  if (tid < 2 * (R0 + 16)) {  // the new rows' columns as operands (2 threads a column)
    const int b = tid >> 1, k0 = 8 * (tid & 1);
    int m = -kBad;
#pragma unroll
    for (int k = 0; k < 8; ++k) m = max(m, shifted(V[(R0 + k0 + k) * LD + b], -hs[R0 + k0 + k]));
    m = max(m, __shfl_xor_sync(~0u, m, 1));
    const int e = row_exp(m);
    if (k0 == 0) sb.ec[48 * Q + b] = e;
#pragma unroll
    for (int k = 0; k < 8; ++k)
      sb.ic[b * kLI + R0 + k0 + k] = halves_of(V[(R0 + k0 + k) * LD + b], -hs[R0 + k0 + k], e);
  }
  bar();
  for (int idx = tid; idx < 16 * (R0 + 16); idx += 128) {
    const int a = idx & 15, b = idx >> 4;
    double s = 0.0;
    for (int M = b >> 4; M <= Q; ++M) {
      IntDot acc;
#pragma unroll 4
      for (int m = 0; m < 16; ++m) acc.add(sa.ia[(R0 + 16 + a) * kLI + 16 * M + m], sb.ic[b * kLI + 16 * M + m]);
      s += scaled_double(acc.value(), sa.ea[64 * M + R0 + 16 + a] + sb.ec[48 * M + b] - 56);
    }
    sb.x[a * 49 + b] = s;
  }
}

// Diagonal block: LDL^T with dynamic regularisation of the pw x pw block at G and the inverse of
// its unit lower factor, left in shared memory: A and V (64 x 65: L with the pivots, L^{-1}); D and
// the scalings gs, hs are written.
//
// bf_diag_block took 113 us here: it is FP64 warp instructions on one SM (64 clocks each, 76 with all
// four sub-partitions busy), many with few active lanes.  Panels of 16 columns on four warps: per
// pivot one column goes through shared memory and one barrier; the reciprocal, the test of
// the sign and the products with 16 terms (the trailing updates, and the off-diagonal blocks of
// L^{-1}) are integer arithmetic, the products exact (operands scaled like the packs).  Warps 4-7
// form L^{-1} a block row behind the panels, and the part of the trailing update that
// the next panel does not read.  64 us with the packs: panels 12 us each, the last row of L^{-1} 5.5.
__device__ int diag64(const double* G, int64_t f, int pw, double* D, const int8_t* dsign, double eps, double delta,
                      double* scr, Diag64Smem& sa, Diag64SmemB& sb, DiagScratch<double>& sh, int* gs, int* hs) {
  constexpr int LD = kDiagLD;
  double* A = scr;
  double* V = scr + 64 * LD;
  const int tid = threadIdx.x, wid = tid >> 5;
  const long long key_eps = order_key(eps + 0.0);
  if (tid < 64) sh.sgn[tid] = tid < pw ? dsign[tid] : (int8_t)1;
  for (int idx = tid; idx < 64 * 64; idx += NT) {
    const int i = idx & 63, j = idx >> 6;
    double v = 0.0;
    if (i < pw && j < pw && i >= j) v = __ldcg(G + i + (int64_t)j * f);
    else if (i == j) v = 1.0;  // rows and pivots past pw: the identity
    A[i * LD + j] = v;
    V[i * LD + j] = 0.0;
    if (i == j) {  // g: half the exponent of the diagonal
      const int lg = i < pw ? ilog_of(v) : 0;
      gs[i] = lg <= -kBad || lg >= kBad ? 0 : lg >> 1;
    }
  }
  const double rdelta = 1.0 / delta;
  __syncthreads();
  int nhit = 0;
  for (int q = 0; q < 4; ++q) {
    if (wid < 4) {
      if (q < 2) diag64_panel<2>(q, pw, A, sa, sb, sh, hs, key_eps, delta, rdelta, nhit);
      else diag64_panel<4>(q, pw, A, sa, sb, sh, hs, key_eps, delta, rdelta, nhit);
    } else if (q > 0) {
      for (int I = q + 1; I < 4; ++I)  // the rest of panel q - 1's update
        for (int J = q + 1; J <= I; ++J) {
          diag64_update(q - 1, I, J, tid - 128, A, sa, sb);
          diag64_update(q - 1, I, J, tid, A, sa, sb);
        }
      diag64_inverse_row(q - 1, tid - 128, A, V, sa, sb, gs, hs);
    }
    __syncthreads();
    for (int I = q + 1; I < 4; ++I) diag64_update(q, I, q + 1, tid, A, sa, sb);
    __syncthreads();
  }
  if (wid >= 4) diag64_inverse_row(3, tid - 128, A, V, sa, sb, gs, hs);
  __syncthreads();
  if (__syncthreads_or(tid < 64 && hs[tid] > gs[tid])) {  // e_k (four threads a row), then g (four a column): see the top
    const int a = tid >> 2, b0 = 16 * (tid & 3);
    int e = -kBad, m = -kBad;
#pragma unroll
    for (int l = b0; l < b0 + 16; ++l) e = max(e, shifted(V[a * LD + l], gs[l]));
    e = max(e, __shfl_xor_sync(~0u, e, 1));
    e = max(e, __shfl_xor_sync(~0u, e, 2));
    if (b0 == 0) sa.xm[a] = max(e, hs[a]);
    __syncthreads();
#pragma unroll
    for (int k = b0; k < b0 + 16; ++k) m = max(m, shifted(V[k * LD + a], -sa.xm[k]));
    m = max(m, __shfl_xor_sync(~0u, m, 1));
    m = max(m, __shfl_xor_sync(~0u, m, 2));
    if (b0 == 0) gs[a] = block_scale(m);
  }
  for (int i = tid; i < pw; i += NT) D[i] = sh.dv[i];
  return nhit;
}

struct Packs {
  unsigned char* base;
  int64_t nL, P, nbf;
  __device__ int64_t l(int p, int64_t i) const {
    return (int64_t)p * (nbf - 1) - (int64_t)p * (p - 1) / 2 + (i - p - 1);
  }
  __device__ unsigned char* pa(int p, int64_t i) const { return base + kTileStride * l(p, i); }
  __device__ unsigned char* pb(int p, int64_t i) const { return base + kTileStride * (nL + l(p, i)); }
  __device__ unsigned char* pe(int p, int64_t e) const { return base + kTileStride * (2 * nL + (int64_t)p * (p + 1) / 2 + e); }
  __device__ unsigned char* pt(int p) const { return base + kTileStride * (2 * nL + P * (P + 1) / 2 + p); }
};
__device__ __forceinline__ int* exps_of(unsigned char* t) { return reinterpret_cast<int*>(t + kPackBytes); }

__global__ void __launch_bounds__(NT, 1)
    k_bf_flow64(BigFrontDev bf, const FlowTask* __restrict__ task, int64_t t0, int64_t nt, int* __restrict__ state,
                int64_t head_off, const int64_t* __restrict__ soff, double* F, double* E, double* Dp,
                const int8_t* __restrict__ dsign, double eps, double delta, int* hits, int* err, const int* skip,
                unsigned char* pk) {
  if (skip && *skip) return;
  extern __shared__ __align__(16) unsigned char smraw[];
  unsigned char* sm = smraw + ((1024u - (s_addr(smraw) & 1023u)) & 1023u);
  unsigned char* smB = sm + kOffB;
  double* scr = reinterpret_cast<double*>(sm + kOffS);
  double* scr2 = scr + kTile;
  __shared__ DiagScratch<double> dsh;
  __shared__ int eA[64], eB[64], hs[64], gs[64];  // row exponents of the operands; h; g
  __shared__ double dinv[64], dinv2[64];  // 1 / d_j and what its rounding left
  __shared__ FlowTask s_task;
  __shared__ int s_go, s_flag;
  __shared__ __align__(8) uint64_t s_bar[2];
  __shared__ uint32_t s_tmem;
  int* head = state + head_off;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(s_addr(&s_bar[0])), "r"(1));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(s_addr(&s_bar[1])), "r"(1));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_flag = 0;
  }
  for (int k = tid; k < kSlice / 16; k += NT) reinterpret_cast<uint4*>(sm + kDig * kSlice)[k] = make_uint4(0, 0, 0, 0);
  if (wid == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_addr(&s_tmem)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  fence_async_shared();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = s_tmem;
  const uint32_t bar_ld = s_addr(&s_bar[0]), bar_mma = s_addr(&s_bar[1]);
  uint32_t par_ld = 0, par_mma = 0;
  // row and columns of this thread's part of a product
  const int orow = 32 * (wid & 1) + lane, ocol = 16 * (2 * (wid >> 2) + ((wid >> 1) & 1));
  for (;;) {
    if (tid == 0) {
      const int cur = atomicAdd(head, 1);
      int go = 0;
      if (cur < nt) {
        const FlowTask tk = task[t0 + cur];
        s_task = tk;
        const int64_t b = tk.bf;
        const Geo g{bf.f[b], bf.c[b], (bf.c[b] + NB - 1) / NB, flow_nbf(bf.f[b], bf.c[b])};
        const Words w = words_of(state + soff[b], g);
        const int p = tk.p;
        const int* wp[3];
        int wv[3];
        int nw;
        switch (tk.kind) {
          case 0:
            wp[0] = w.t(p, p), wv[0] = p;
            nw = 1;
            break;
          case 1:
            wp[0] = w.diag + p, wv[0] = 1;
            wp[1] = w.t(tk.i, p), wv[1] = p;
            nw = 2;
            break;
          case 2:
            wp[0] = w.diag + p, wv[0] = 1;
            wp[1] = w.e(p, tk.j), wv[1] = p - tk.j;
            nw = 2;
            break;
          case 3:
            wp[0] = w.trsm + tk.i, wv[0] = p + 1;
            wp[1] = w.trsm + tk.j, wv[1] = p + 1;
            wp[2] = w.t(tk.i, tk.j), wv[2] = p;
            nw = 3;
            break;
          default:
            wp[0] = w.trsm + tk.i, wv[0] = p + 1;
            if (tk.j < p)
              wp[1] = w.e(p, tk.j), wv[1] = p - tk.j + 1;
            else
              wp[1] = w.pe + p, wv[1] = 1;
            wp[2] = w.e(tk.i, tk.j), wv[2] = p - tk.j;
            nw = 3;
            break;
        }
        int got[3] = {0, 0, 0};
#pragma unroll
        for (int q = 0; q < 3; ++q)
          if (q < nw) got[q] = ld_relaxed(wp[q]);
        bool ok = true;
#pragma unroll
        for (int q = 0; q < 3; ++q)
          if (q < nw && got[q] < wv[q]) ok = ok && wait_ge(wp[q], wv[q], err);
        go = ok ? 1 : 0;
        if (ok) __threadfence();
      }
      s_go = go;
    }
    __syncthreads();
    if (!s_go) break;
    const FlowTask tk = s_task;
    const int64_t b = tk.bf;
    const Geo g{bf.f[b], bf.c[b], (bf.c[b] + NB - 1) / NB, flow_nbf(bf.f[b], bf.c[b])};
    const Packs pkr{pk + (int64_t)kTileStride * bf.pkoff64[b], flow_pk_nl(g.f, g.c), g.P, g.nbf};
    const Words w = words_of(state + soff[b], g);
    const int p = tk.p, pw = bnrow(g, p);
    const int64_t f = g.f, k0 = (int64_t)p * NB;
    double* G = F + bf.goff[b];
    double* Eb = E + bf.eoff[b];
    const int64_t kp = bf.k0pos[b] + k0;
    bool stop = false;
    // a task's products: copies of the packs (thread 0), then, with the A digits in place, the MMAs
    auto wait_bar = [&](uint32_t bar, uint32_t& par) {
      if (!mbar_wait(bar, par)) atomicExch(&s_flag, 1);
      __syncthreads();
      if (s_flag) {
        if (tid == 0) {
          atomicExch(err, 2);
          mbar_wait(bar, par);  // once more for the copies or MMAs in flight
        }
        return false;
      }
      par ^= 1u;
      return true;
    };
    if (tk.kind == 0) {
      // D(p): the diagonal block on the FP64 pipe, then its packs
      const int nhit = diag64(G + k0 + k0 * f, f, pw, Dp + kp, dsign + kp, eps, delta, scr,
                              *reinterpret_cast<Diag64Smem*>(sm), *reinterpret_cast<Diag64SmemB*>(smB), dsh, gs, hs);
      if (tid == 0 && nhit) atomicAdd(hits, nhit);
      __syncthreads();
      if (tid < 64) {
        int* ex = exps_of(pkr.pt(p));
        ex[64 + tid] = gs[tid];
        ex[128 + tid] = hs[tid];
      }
      const double* V = scr + 64 * kDiagLD;
      pack_tile(V, kDiagLD, 1, 0, gs, 1, pkr.pt(p), exps_of(pkr.pt(p)));
      fence_async_global();
      __syncthreads();
      if (tid == 0) {
        __threadfence();
        st_release(w.diag + p, 1);
      }
      // after the release: what no T(p, i) or Efin(p, e) reads: L_KK and its inverse for the solves, and
      // PE(p, p), rows the columns of Linv, for EU(p, i, p)
      pack_tile(V, 1, kDiagLD, 0, hs, -1, pkr.pe(p, p), exps_of(pkr.pe(p, p)));
      fence_async_global();
      fence_async_shared();  // the operands' space is the next task's, by bulk copies
      __syncthreads();
      if (tid == 0) {
        __threadfence();
        st_release(w.pe + p, 1);
      }
      for (int idx = tid; idx < 64 * 64; idx += NT) {
        const int i = idx & 63, j = idx >> 6;
        if (i < pw && j < pw && i >= j) {
          G[(k0 + i) + (k0 + j) * f] = scr[i * kDiagLD + j];
          Eb[(k0 + i) + (k0 + j) * f] = (i == j) ? 1.0 : V[i * kDiagLD + j];
        }
      }
      __syncthreads();
      continue;
    }
    // T(p, i): rows of F_IK; Efin(p, e): rows the columns of E_KC; both times PT(p)^T.  U(p, i, j),
    // EU(p, i, e): PA(p, i) times PB(p, j)^T or PE(p, e)^T
    const bool upd = tk.kind >= 3, efin = tk.kind == 2, etile = tk.kind == 4;
    const int64_t i0 = efin ? (int64_t)tk.j * NB : brow0(g, tk.i), c0 = etile ? (int64_t)tk.j * NB : brow0(g, tk.j);
    const int ni = efin ? NB : bnrow(g, tk.i), nc = bnrow(g, tk.j);
    const bool diag = tk.kind == 3 && tk.i == tk.j;
    double* base = etile ? Eb : G;
    unsigned char* tb = !upd ? pkr.pt(p) : (etile ? pkr.pe(p, tk.j) : pkr.pb(p, tk.j));
    if (tid == 0) {
      fence_async_global();  // the packs were stored by generic writes (acquired above)
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar_ld),
                   "r"((upd ? 2 : 1) * kPackBytes)
                   : "memory");
      if (upd) bulk_copy(s_addr(sm), pkr.pa(p, tk.i), kPackBytes, bar_ld);
      bulk_copy(s_addr(smB), tb, kPackBytes, bar_ld);
    }
    if (tid < 64) eB[tid] = __ldcg(exps_of(tb) + tid);
    double tv[16];
    if (upd) {
      if (tid >= 64 && tid < 128) eA[tid - 64] = __ldcg(exps_of(pkr.pa(p, tk.i)) + tid - 64);
#pragma unroll
      for (int u = 0; u < 16; ++u) {
        const int cc = ocol + u;
        tv[u] = (orow < ni && cc < nc && (!diag || orow >= cc)) ? __ldcg(base + (i0 + orow) + (c0 + cc) * f) : 0.0;
      }
    } else {
      if (tid < 64) {
        const int* ex = exps_of(tb);
        gs[tid] = __ldcg(ex + 64 + tid);
        hs[tid] = __ldcg(ex + 128 + tid);
      } else if (tid < 128 && !efin) {
        const int k = tid - 64;
        const double d = k < pw ? __ldcg(Dp + kp + k) : 1.0, r = 1.0 / d;
        dinv[k] = k < pw ? r : 0.0;
        dinv2[k] = k < pw ? fma(-d, r, 1.0) * r : 0.0;
      }
      // the tile: lane along the rows of F, or along k (the rows of E)
      const int a = tid & 63, b0 = tid >> 6;
      double x[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) {
        const int c = b0 + 4 * u, r = efin ? c : a, k = efin ? a : c;
        x[u] = (r < ni && k < pw) ? __ldcg(efin ? Eb + (k0 + k) + (i0 + r) * f : G + (i0 + r) + (k0 + k) * f) : 0.0;
      }
#pragma unroll
      for (int u = 0; u < 16; ++u) {
        const int c = b0 + 4 * u;
        scr[efin ? tile_at(a) + c : tile_at(c) + a] = x[u];
      }
      __syncthreads();
      pack_tile(scr, 1, 65, 8, gs, -1, sm, eA);
      fence_async_shared();
    }
    stop = !wait_bar(bar_ld, par_ld);
    if (!stop) {
      if (tid == 0) issue_products(s_addr(sm), s_addr(smB), tmem, bar_mma);
      stop = !wait_bar(bar_mma, par_mma);
    }
    if (stop) break;
    read_products(tmem, eA, eB, scr, scr2);
    if (upd) {
#pragma unroll
      for (int u = 0; u < 16; ++u) {
        const int cc = ocol + u;
        if (orow < ni && cc < nc && (!diag || orow >= cc))
          base[(i0 + orow) + (c0 + cc) * f] = tv[u] - scr[tile_at(cc) + orow];
      }
    } else if (efin) {
      const int a = tid & 63;
      if (a < pw)
#pragma unroll 4
        for (int c = tid >> 6; c < NB; c += 4) Eb[(k0 + a) + (i0 + c) * f] = scr[tile_at(a) + c];
    } else {
      const int a = tid & 63;
#pragma unroll 4
      for (int c = tid >> 6; c < NB; c += 4) {
        const bool in = c < pw && a < ni;
        const double o = in ? scr[tile_at(c) + a] : 0.0, q = fma(o, dinv[c], o * dinv2[c]);  // o / d to half an ulp
        if (in) G[(i0 + a) + (k0 + c) * f] = q;
        if (!in) scr[tile_at(c) + a] = 0.0;
        scr2[tile_at(c) + a] = q;
      }
      __syncthreads();
      pack_tile(scr2, 1, 65, 8, hs, 1, pkr.pa(p, tk.i), exps_of(pkr.pa(p, tk.i)));
    }
    if (!upd) {
      unsigned char* dst = efin ? pkr.pe(p, tk.j) : pkr.pb(p, tk.i);
      pack_tile(scr, 1, 65, 8, hs, -1, dst, exps_of(dst));
      fence_async_global();
    }
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      if (tk.kind == 1) st_release(w.trsm + tk.i, p + 1);
      else if (tk.kind == 2) st_release(w.e(p, tk.j), p - (int)tk.j + 1);
      else if (etile) st_release(w.e(tk.i, tk.j), p - (int)tk.j + 1);
      else st_release(w.t(tk.i, tk.j), p + 1);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (wid == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}
}  // namespace

int flow64_setup_attributes() {
  CLR_CUDA(cudaFuncSetAttribute(k_bf_flow64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem));
  return CLR_OK;
}

int flow64_level(cudaStream_t st, const BigFrontDev& bf, const FlowTask* task, int64_t t0, int64_t nt, int* state,
                 int64_t head_off, const int64_t* soff, int grid, double* F, double* E, double* Dp, const int8_t* dsign,
                 double eps, double delta, int* hits, int* err, const int* skip, unsigned char* pk) {
  if (nt <= 0) return CLR_OK;
  k_bf_flow64<<<(unsigned)std::min<int64_t>(nt, grid), NT, kSmem, st>>>(bf, task, t0, nt, state, head_off, soff, F, E, Dp,
                                                                       dsign, eps, delta, hits, err, skip, pk);
  CLR_CHECK_LAUNCH();
  return CLR_OK;
}

}  // namespace clr
