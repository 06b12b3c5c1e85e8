// The epilogue of the narrow-layer kernels (k_pw_conv.cu, k_c3_conv.cu): one
// warp takes the 32 accumulator rows of its TMEM lane quarter and up to 64
// columns at a time -- the accumulator in one or two wide TMEM loads, the second
// operand X (forward: the residual, data gradient: the BN input) from shared
// memory, the output staged in one swizzled tile and stored by TMA through a
// Dst, the column sums from the staged tile with two columns a lane.
#pragma once
#include "pnn_internal.h"
#include "tc_pair.cuh"
#include "tc_ptx.cuh"

namespace pnn {
namespace tc {

enum { FWD = 0, DGRAD = 1 };
constexpr int kRedBytes = 2 * 4 * 64 * 8;  // per epilogue group: [2][4 warps][64 columns] pairs
// per-warp output staging: forward one 32 x 64 bf16 tile, data gradient two of 32 x 32 fp32
__host__ __device__ constexpr int stage_bytes(int mode) { return mode == FWD ? 4096 : 8192; }

// whether a unit has a second operand: the residual (forward), the BN input
// of the sums (data gradient)
template <int MODE>
__device__ __forceinline__ bool has_x(const ConvDesc* d) {
  return MODE == FWD ? d->res != nullptr : d->bnb_part != nullptr;
}

// byte offset of 16-byte chunk j of a row in a TMA-swizzled tile of PITCH-byte rows
template <int PITCH>
__device__ __forceinline__ uint32_t swp(int row, int j) {
  if (PITCH == 128) return (uint32_t)(row * 128 + ((j ^ (row & 7)) << 4));
  if (PITCH == 64) return (uint32_t)(row * 64 + ((j ^ ((row >> 1) & 3)) << 4));
  return (uint32_t)(row * 32 + ((j ^ ((row >> 2) & 1)) << 4));
}

// what the epilogue needs of an instance, read once an instance
struct EpiArgs {
  const void* y;                                // output map
  float* part;                                  // column partials (or null)
  const float *scale, *shift, *mean, *rstd;     // data gradient: the BN of the sums
  bool stats, hx, acc, relu;
  template <int MODE>
  __device__ __forceinline__ void load(const ConvDesc* d) {
    y = d->tma_y;
    part = MODE == FWD ? d->stats : d->bnb_part;
    stats = part != nullptr;
    hx = has_x<MODE>(d);
    acc = MODE == DGRAD && d->accumulate;
    if (MODE == DGRAD) {
      scale = d->x.scale;
      shift = d->x.shift;
      mean = d->bn_mean;
      rstd = d->bn_rstd;
      relu = d->x.relu != 0;
    }
  }
};

struct EpiState {
  float2* red;  // this group's [2][4][64] pairs
  int rbuf;     // which half the next unit uses
  int bar;      // the group's named barrier
};

// The four warps' column pairs of a unit -> the tile's partial: forward (mean,
// M2) merged in order, data gradient plain sums.  Every warp of the group
// calls it (ok: its own values are valid); one barrier, the halves of red
// alternate.
template <int MODE, int BN>
__device__ __forceinline__ void merge_partials(EpiState& es, bool ok, int q, int lane, int rows, int m0, float* part) {
  float2* red = es.red + es.rbuf * 256;
  es.rbuf ^= 1;
  asm volatile("bar.sync %0, 128;" ::"r"(es.bar) : "memory");
  const int j = q * 32 + lane;
  if (j < BN && ok) {
    float a, b;
    if (MODE == FWD) {
      float n = 0.f;
      a = b = 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int nq = min(32, max(0, rows - (m0 + 32 * i)));
        const float2 v = red[i * 64 + j];
        chan_merge(n, a, b, (float)nq, v.x, v.y);
      }
    } else {
      const float2 v0 = red[j], v1 = red[64 + j], v2 = red[128 + j], v3 = red[192 + j];
      a = v0.x + v1.x + v2.x + v3.x;
      b = v0.y + v1.y + v2.y + v3.y;
    }
    *reinterpret_cast<float2*>(part + 2 * j) = make_float2(a, b);
  }
}

// (mean, M2) of the columns of a staged bf16 tile [32][BN] over its first
// nvalid rows: lane = column pair l % (BN/2) of rows (l / (BN/2)) + RG i, two
// passes (the sums, then the squared deviations from the warp mean)
template <int BN, bool FULL>
__device__ __forceinline__ void staged_moments(const uint8_t* st, int lane, int nvalid, float2* out) {
  constexpr int PITCH = BN * 2, PAIRS = BN / 2, RG = 32 / PAIRS, IT = 32 / RG;
  const int p = lane % PAIRS, g = lane / PAIRS;
  uint32_t w[IT];
#pragma unroll
  for (int i = 0; i < IT; ++i)
    w[i] = *reinterpret_cast<const uint32_t*>(st + swp<PITCH>(RG * i + g, p >> 2) + (p & 3) * 4);
  uint64_t s[2] = {0ull, 0ull};
#pragma unroll
  for (int i = 0; i < IT; ++i) {
    if (!FULL && RG * i + g >= nvalid) w[i] = 0u;
    s[i & 1] = add2(s[i & 1], bf2(w[i]));
  }
  float2 sum = un2(add2(s[0], s[1]));
#pragma unroll
  for (int o = PAIRS; o < 32; o <<= 1) {
    sum.x += __shfl_xor_sync(0xffffffffu, sum.x, o);
    sum.y += __shfl_xor_sync(0xffffffffu, sum.y, o);
  }
  const float n = (float)nvalid;
  const float mx = FULL ? sum.x * 0.03125f : (nvalid > 0 ? sum.x / n : 0.f);
  const float my = FULL ? sum.y * 0.03125f : (nvalid > 0 ? sum.y / n : 0.f);
  const uint64_t neg = pk2(-mx, -my);
  s[0] = s[1] = 0ull;
#pragma unroll
  for (int i = 0; i < IT; ++i) {
    const uint64_t d = add2(bf2(w[i]), neg);
    if (FULL || RG * i + g < nvalid) s[i & 1] = fma2(d, d, s[i & 1]);
  }
  float2 m2 = un2(add2(s[0], s[1]));
#pragma unroll
  for (int o = PAIRS; o < 32; o <<= 1) {
    m2.x += __shfl_xor_sync(0xffffffffu, m2.x, o);
    m2.y += __shfl_xor_sync(0xffffffffu, m2.y, o);
  }
  if (g == 0) *reinterpret_cast<float4*>(out + 2 * p) = make_float4(mx, m2.x, my, m2.y);
}

// Forward unit: accumulator + residual -> bf16 -> staging -> TMA store, statistics.
template <int BN, typename Dst>
__device__ __forceinline__ void unit_fwd(const EpiArgs& ea, const Dst& dst, uint32_t tacc, int q, int lane, int rows, int m0, int n0,
                                         const uint8_t* x, uint8_t* st, float2* redw, uint32_t tempty,
                                         uint32_t uempty, bool leader) {
  uint32_t a[BN];
#pragma unroll
  for (int j = 0; j < BN; j += 32) {
    if (BN >= 32) tmem_ld32(tacc + j, a + j);
    else tmem_ld16_nowait(tacc + j, a + j);
  }
  tmem_wait_ld(a);
  fence_before();
  __syncwarp();
  if (lane == 0) mbar_arrive(tempty);
  constexpr int PITCH = BN * 2;
  uint32_t o[BN / 2];
  if (ea.hx) {
#pragma unroll
    for (int j = 0; j < BN / 8; ++j) {
      const uint4 r = *reinterpret_cast<const uint4*>(x + swp<PITCH>(q * 32 + lane, j));
      const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int c = 8 * j + 2 * i;
        o[4 * j + i] = pack2(add2(pk2(__uint_as_float(a[c]), __uint_as_float(a[c + 1])), bf2(w[i])));
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < BN / 2; ++i) o[i] = pack_bf16(__uint_as_float(a[2 * i]), __uint_as_float(a[2 * i + 1]));
  }
  // the store issued from this tile for the previous unit must have read it,
  // and every lane must be done with its statistics
  if (leader) bulk_wait_read<0>();
  __syncwarp();
  if (ea.hx && lane == 0) mbar_arrive(uempty);  // X has been read
#pragma unroll
  for (int j = 0; j < BN / 8; ++j)
    *reinterpret_cast<uint4*>(st + swp<PITCH>(lane, j)) = make_uint4(o[4 * j], o[4 * j + 1], o[4 * j + 2], o[4 * j + 3]);
  fence_proxy_async();
  __syncwarp();
  const int nvalid = min(32, max(0, rows - (m0 + q * 32)));
  if (leader && nvalid > 0) {
    dst.put(ea.y, n0, q, smem_u32(st), false);
    bulk_commit();
  }
  if (ea.stats) {
    if (nvalid == 32) staged_moments<BN, true>(st, lane, 32, redw);
    else staged_moments<BN, false>(st, lane, nvalid, redw);
  }
}

// BN-backward sums of HC columns of a staged dX tile [32][HC] fp32 with the
// unit's h tile [128][BN] bf16: g = dX masked by the ReLU of the forward BN
// output, xhat = (h - mean) * rstd; (sum g, sum g xhat) over the valid rows.
template <int BN, bool FULL>
__device__ __forceinline__ void staged_bn_sums(const uint8_t* st, const uint8_t* h, int c0, const EpiArgs& ea, int n0, int q,
                                               int lane, int nvalid, float2* out) {
  constexpr int HC = BN < 32 ? BN : 32;
  constexpr int PAIRS = HC / 2, RG = 32 / PAIRS, IT = 32 / RG;
  const int p = lane % PAIRS, g = lane / PAIRS;
  const int c = n0 + c0 + 2 * p;
  const float2 scv = __ldg(reinterpret_cast<const float2*>(ea.scale + c));
  const float2 shv = __ldg(reinterpret_cast<const float2*>(ea.shift + c));
  const float2 muv = __ldg(reinterpret_cast<const float2*>(ea.mean + c));
  const float2 rsv = __ldg(reinterpret_cast<const float2*>(ea.rstd + c));
  const uint64_t sc = pk2(scv.x, scv.y), sh = pk2(shv.x, shv.y), nmu = pk2(-muv.x, -muv.y), rs = pk2(rsv.x, rsv.y);
  const bool relu = ea.relu;
  uint64_t s1 = 0ull, s2 = 0ull;
#pragma unroll
  for (int i = 0; i < IT; ++i) {
    // rows r and r + 4 of 128-byte h rows fall into different halves of the banks
    const int r = BN == 64 ? (i & 3) + 8 * (i >> 2) + 4 * g : RG * i + g;
    const int hc = c0 / 2 + p;
    const uint32_t hw =
        *reinterpret_cast<const uint32_t*>(h + swp<BN * 2>(q * 32 + r, hc >> 2) + (hc & 3) * 4);
    const float2 dv = *reinterpret_cast<const float2*>(st + swp<HC * 4>(r, p >> 1) + (p & 1) * 8);
    const uint64_t hv = bf2(hw);
    const float2 z = un2(fma2(sc, hv, sh));
    const bool in = FULL || r < nvalid;
    const uint64_t gv = pk2(in && (!relu || z.x > 0.f) ? dv.x : 0.f, in && (!relu || z.y > 0.f) ? dv.y : 0.f);
    const uint64_t xh = mul2(add2(hv, nmu), rs);
    s1 = add2(s1, gv);
    // (a row past the end adds nothing: its h may be anything)
    if (in) s2 = fma2(gv, xh, s2);
  }
  float2 a = un2(s1), b = un2(s2);
#pragma unroll
  for (int o = PAIRS; o < 32; o <<= 1) {
    a.x += __shfl_xor_sync(0xffffffffu, a.x, o);
    a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
    b.x += __shfl_xor_sync(0xffffffffu, b.x, o);
    b.y += __shfl_xor_sync(0xffffffffu, b.y, o);
  }
  if (g == 0) *reinterpret_cast<float4*>(out + c0 + 2 * p) = make_float4(a.x, b.x, a.y, b.y);
}

// Data-gradient unit: accumulator -> fp32 staging -> TMA store or reduce-add, BN-backward sums.
template <int BN, typename Dst>
__device__ __forceinline__ void unit_dgrad(const EpiArgs& ea, const Dst& dst, uint32_t tacc, int q, int lane, int rows, int m0, int n0,
                                           const uint8_t* h, uint8_t* stage, int& sbuf, float2* redw, uint32_t tempty,
                                           uint32_t uempty, bool leader) {
  constexpr int HC = BN < 32 ? BN : 32;
  const int nvalid = min(32, max(0, rows - (m0 + q * 32)));
#pragma unroll
  for (int c0 = 0; c0 < BN; c0 += HC) {
    uint32_t a[HC];
    if (HC == 32) tmem_ld32(tacc + c0, a);
    else tmem_ld16_nowait(tacc + c0, a);
    tmem_wait_ld(a);
    if (c0 + HC >= BN) {
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty);
    }
    // the store issued from this buffer two turns ago must have read it: every turn
    // commits a group, an empty one where the warp's rows lie past the layer's end
    if (leader) bulk_wait_read<1>();
    __syncwarp();
    uint8_t* st = stage + sbuf * 4096;
    sbuf ^= 1;
#pragma unroll
    for (int j = 0; j < HC / 4; ++j)
      *reinterpret_cast<uint4*>(st + swp<HC * 4>(lane, j)) = make_uint4(a[4 * j], a[4 * j + 1], a[4 * j + 2], a[4 * j + 3]);
    fence_proxy_async();
    __syncwarp();
    if (leader) {
      if (nvalid > 0) dst.put(ea.y, n0 + c0, q, smem_u32(st), ea.acc);
      bulk_commit();
    }
    if (ea.stats) {
      if (nvalid == 32) staged_bn_sums<BN, true>(st, h, c0, ea, n0, q, lane, 32, redw);
      else staged_bn_sums<BN, false>(st, h, c0, ea, n0, q, lane, nvalid, redw);
    }
  }
  __syncwarp();
  if (ea.stats && lane == 0) mbar_arrive(uempty);  // h has been read
}

}  // namespace tc
}  // namespace pnn
