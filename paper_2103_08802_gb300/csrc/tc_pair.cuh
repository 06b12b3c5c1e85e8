// Shared pieces of the persistent warp-specialised kernels (k_pw_conv.cu,
// k_wg_conv.cu): packed fp32 pairs, wide TMEM loads, ring cursors and the walk
// over a launch's items.
#pragma once
#include "pnn_internal.h"
#include "tc_ptx.cuh"

namespace pnn {
namespace tc {

// position in a ring of n slots and the parity of its current lap
struct Cursor {
  int n, s;
  uint32_t ph;
  __device__ __forceinline__ explicit Cursor(int slots) : n(slots), s(0), ph(0) {}
  __device__ __forceinline__ void next() {
    if (++s == n) { s = 0; ph ^= 1; }
  }
};

__device__ __forceinline__ uint64_t pk2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 un2(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// the two bf16 of a word as an fp32 pair
__device__ __forceinline__ uint64_t bf2(uint32_t w) {
  return pk2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}
__device__ __forceinline__ uint32_t pack2(uint64_t v) {
  const float2 f = un2(v);
  return pack_bf16(f.x, f.y);
}
// max(v, 0) of both bf16 (a NaN becomes 0, as fmaxf(v, 0) makes it)
__device__ __forceinline__ uint32_t relu2(uint32_t w) {
  uint32_t r;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(w), "r"(0u));
  return r;
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,"
      "%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
// wait for this thread's TMEM loads; the registers pass through, so no use of
// them can be scheduled before it
template <int N>
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&r)[N]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < N; i += 8)
    asm volatile("" : "+r"(r[i]), "+r"(r[i + 1]), "+r"(r[i + 2]), "+r"(r[i + 3]), "+r"(r[i + 4]), "+r"(r[i + 5]),
                      "+r"(r[i + 6]), "+r"(r[i + 7]));
}

// Walks the items of one CTA (blockIdx.x, + gridDim.x, ...).  Instances are
// found by stepping forward, so an item costs no division and no descriptor
// reload unless the instance changes.
struct Walk {
  int item, total, inst, t0, t1;         // instance inst owns items t0 .. t1 - 1
  int tm, tn, mt;                        // m-tile and N item within the instance, its m-tiles
  bool fresh;                            // the instance changed with this item
  const ConvDesc* d;
  __device__ __forceinline__ Walk(const ConvDesc* tab, const int* ts, int tot) {
    item = blockIdx.x;
    total = tot;
    inst = -1;
    t0 = 0;
    t1 = 0;
    tm = tn = mt = 0;
    fresh = false;
    d = nullptr;
    settle(tab, ts);
  }
  __device__ __forceinline__ bool more() const { return item < total; }
  __device__ __forceinline__ void settle(const ConvDesc* tab, const int* ts) {
    if (item >= total) return;
    if (item >= t1) {
      do {
        ++inst;
        t0 = t1;
        t1 = __ldg(ts + inst + 1);
      } while (item >= t1);
      d = tab + inst;
      mt = __ldg(&d->mtiles);
      tm = item - t0;
      tn = 0;
      fresh = true;
    } else {
      tm += gridDim.x;
      fresh = false;
    }
    while (tm >= mt) { tm -= mt; ++tn; }
  }
  __device__ __forceinline__ void next(const ConvDesc* tab, const int* ts) {
    item += gridDim.x;
    settle(tab, ts);
  }
};

}  // namespace tc
}  // namespace pnn
