// Version words, bounded waits and geometry of the dataflow factorization kernels.
#pragma once

#include "bigfront.cuh"

namespace clr {
namespace {
constexpr uint32_t kSpin = 1u << 21;  // polls of one wait (about 2 s) before it gives up

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ int ld_relaxed(const int* p) {
  int v;
  asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(int* p, int v) {
  asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Thread 0: wait until *p >= v.  False if the wait ran out (err := 2) or another
// CTA has given up (err != 0).
__device__ bool wait_ge(const int* p, int v, int* err) {
  for (uint32_t it = 0; it < kSpin; ++it) {
    if (ld_acquire(p) >= v) return true;
    if (it >= 16) {
      if (ld_acquire(err) != 0) return false;
      __nanosleep(64);
    }
  }
  atomicExch(err, 2);
  return false;
}

struct Geo {
  int64_t f, c, P, nbf;
};
__device__ __forceinline__ int64_t brow0(const Geo& g, int64_t b) { return b < g.P ? kBfNB * b : g.c + kBfNB * (b - g.P); }
__device__ __forceinline__ int bnrow(const Geo& g, int64_t b) {
  return (int)(b < g.P ? min((int64_t)kBfNB, g.c - kBfNB * b) : min((int64_t)kBfNB, g.f - g.c - kBfNB * (b - g.P)));
}
struct Words {
  int *tile, *etile, *diag, *trsm, *pe, *txc, *uxc;
  int64_t P;
  __device__ int* t(int64_t i, int64_t j) const { return tile + i * (i + 1) / 2 + j; }
  __device__ int* e(int64_t i, int64_t c) const { return etile + i * P + c; }
};
__device__ __forceinline__ Words words_of(int* base, const Geo& g) {
  Words w;
  w.P = g.P;
  w.tile = base;
  w.etile = base + g.nbf * (g.nbf + 1) / 2;
  w.diag = w.etile + g.nbf * g.P;
  w.trsm = w.diag + g.P;
  w.pe = w.trsm + g.nbf;
  w.txc = w.pe + g.P;
  w.uxc = w.txc + g.P;
  return w;
}

// bounded wait on an mbarrier phase (false: it ran out)
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  for (uint32_t it = 0; it < (1u << 22); ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,"
      "%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
        "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
}  // namespace
}  // namespace clr
