// Grouped weight gradients of stride-1 layers, 1x1 with few channels on one side
// and 3x3, on the 5th-generation tensor cores:
//
//   dW[k][r][s][c] = sum_{pixels p} dY[p][k] * act(X)[p + (r-1, s-1)][c]
//
// The contraction runs over pixels, so both operands keep a pixel's channels
// together as they arrive (MN-major): no-swizzle planes of 16-byte pixel rows,
// one plane per 8 channels.  Every element is transformed once (activation:
// BN scale/shift + ReLU of the producing layer, bf16; gradient: bf16) and
// stored once:
//   1x1   the side with more channels is the MMA's M side (planes past its
//         channels are read but their accumulator rows are not), the other N;
//   3x3   a k-step is R whole image rows; the activation rows y0 - 1 .. y0 + R
//         are stored three times, shifted by one column each way (zero where the
//         tap leaves the row), so the N side of an MMA is three taps at once and
//         the three tap rows are descriptor offsets of one image row.  An MMA
//         costs the read of its M side (128 rows x 16 pixels, 4 KB of shared
//         memory) whatever its N, so nine MMAs of one tap each (one copy with
//         zero columns at its sides) took 146 us where three took 67.
//         (Copying the transformed halo to a plane per tap, as the kernel of
//         k_tc_conv.cu does, took 80 % of that kernel's 224 us.)  Whole images of
//         at most 32 pixels have no rows at a uniform distance: theirs are stored
//         nine times, once a tap.  A tile is a block of 32 by 128 channels: its
//         nine accumulators of 32 columns fit the tensor memory once.
// Plane pitches are padded so that the eight lanes of a 16-byte store phase
// fall into different banks whatever the channel count.
//
// Persistent; a tile is one run of pixels of one instance (and, 3x3, one block
// of its channels): the planner cuts the launch into about
// two tiles per SM of equal traffic, so few partial sums are written and
// reduced.  Roles: producer (TMA, one thread), MMA (one thread), ten transform
// warps, four epilogue warps.  Grouped launches of the
// 8-subnetwork ResNet-1001 (batch 256, 64 px), kernels of k_tc_conv.cu -> now:
// 3x3 224 -> 59 us, expand (16 -> 64) 159 -> 63 us (two launches before), reduce
// 141 -> 52 us; the 1x1 are at 0.68 - 0.84 of the copy rate, the 3x3 is bound by
// the latency of its k-steps.  VGG-16 (batch 128): 128 -> 128 at 16 x 16, 4
// instances, 348 -> 76 us; 256 -> 256 at 8 x 8, 3 instances, 232 -> 68; 512 -> 512
// at 4 x 4 90 -> 55: each block of 32 input channels transforms the gradient again.
// Every wait is bounded (2 s); on expiry the CTA records status 3, stops,
// drains its copies and MMAs (bounded) and frees its TMEM.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "pnn.h"
#include "pnn_internal.h"
#include "tc_pair.cuh"
#include "tc_ptx.cuh"

namespace pnn {
namespace {

using namespace tc;

constexpr int kT = 10, kE = 4;
constexpr int kProducer = 0, kMma = 1, kT0 = 2, kE0 = kT0 + kT;
constexpr int kThreads = 32 * (2 + kT + kE);
constexpr int kNT = 32 * kT;
static_assert(kE0 % 4 == 0, "epilogue warps start at a TMEM lane quarter");
constexpr int kMaxRing = 4;
constexpr int kTmemCols = 512;
constexpr int kSmemBudget = 227 * 1024;
// an A operand's 16 M groups are always read: this much memory follows the operand ring
constexpr int kMReach = 16 * (128 + 8) * 16;  // (a multiple of 1024)

struct Shared {
  uint64_t raw_full[kMaxRing], raw_empty[kMaxRing];
  uint64_t op_full[kMaxRing], op_empty[kMaxRing];
  uint64_t tfull[2], tempty[2];
  uint64_t drain;
  uint32_t tmem;
  int abort_flag;
};

struct Rings {
  int nr, no, rawb, opb;
};
__host__ __device__ inline int rings_raw(const Rings& r) { return r.nr * r.rawb > kMReach ? r.nr * r.rawb : kMReach; }
__host__ __device__ inline int rings_bytes(const Rings& r) { return r.no * r.opb + rings_raw(r); }
constexpr int kFixed = 1024 + (int)sizeof(Shared);

bool plan_rings(int rawb, int opb, Rings& r) {
  r = Rings{2, 2, rawb, opb};
  if (rings_bytes(r) > kSmemBudget - kFixed) return false;
  for (int* n : {&r.nr, &r.no, &r.nr, &r.no}) {
    ++*n;
    if (rings_bytes(r) > kSmemBudget - kFixed) --*n;
  }
  return true;
}

// what the roles need of an instance
struct Geo {
  WgPlan p;
  int C, K, W, H, rows;
  bool xbf, bn;
};
template <int KS>
__device__ __forceinline__ Geo geo(const ConvDesc* d) {
  Geo g;
  g.C = d->C;
  g.K = d->K;
  g.W = d->W;
  g.H = d->H;
  g.rows = d->B * d->H * d->W;
  g.xbf = d->x.dt == DT_BF16;
  g.bn = d->x.scale != nullptr;
  g.p = wg_plan(KS, d->C, d->K, d->H, d->W, g.xbf);
  return g;
}

// ------------------------------------------------------------ transform
// A thread keeps one 8-channel chunk for a whole tile: its BN scale and shift
// stay in registers.
struct Affine {
  uint64_t sc[4], sf[4];
  __device__ __forceinline__ void load(const float* s, const float* f, int c) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 a = __ldg(reinterpret_cast<const float2*>(s + c) + i);
      const float2 b = __ldg(reinterpret_cast<const float2*>(f + c) + i);
      sc[i] = pk2(a.x, a.y);
      sf[i] = pk2(b.x, b.y);
    }
  }
};

// 8 raw elements (bf16: one 16-byte word, fp32: two) -> 8 bf16
template <bool XBF, bool BN>
__device__ __forceinline__ uint4 chunk8(const uint4 (&q)[2], const Affine& af, int relu) {
  uint32_t o[4];
  if (XBF) {
    const uint32_t w[4] = {q[0].x, q[0].y, q[0].z, q[0].w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      o[i] = BN ? pack2(fma2(af.sc[i], bf2(w[i]), af.sf[i])) : w[i];
      if (BN && relu) o[i] = relu2(o[i]);
    }
  } else {
    const uint32_t w[8] = {q[0].x, q[0].y, q[0].z, q[0].w, q[1].x, q[1].y, q[1].z, q[1].w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint64_t v = pk2(__uint_as_float(w[2 * i]), __uint_as_float(w[2 * i + 1]));
      o[i] = BN ? pack2(fma2(af.sc[i], v, af.sf[i])) : pack2(v);
      if (BN && relu) o[i] = relu2(o[i]);
    }
  }
  return make_uint4(o[0], o[1], o[2], o[3]);
}

// Rows of one source: raw [nrows][8 << lg channels] -> planes.  HALO 1: row u is
// pixel u of whole image rows of 1 << lgw pixels, zero unless ylo <= u >> lgw <
// yhi; copy s (2^lg planes after copy s - 1) holds at column x the pixel x + s - 1
// of its row or zero -- the pixel that falls out of the row at one end marks the
// zero at the other.  HALO 2: whole images of 1 << (lgw + ylo) pixels, the same in
// both directions, copy 3 r + s for tap (r, s).
template <bool XBF, bool BN, int HALO>
__device__ __forceinline__ void rows_to_planes(const uint8_t* __restrict__ raw, uint8_t* __restrict__ pl, int nrows,
                                               int lg, int pitch, int t, const Affine& af, int relu, int lgw, int ylo,
                                               int yhi) {
  const int cc = t & ((1 << lg) - 1);
  const int step = kNT >> lg;
  const int rp = (XBF ? 16 : 32) << lg;
  const uint8_t* src = raw + cc * (XBF ? 16 : 32);
  uint8_t* dst = pl + cc * pitch;
  for (int r = t >> lg; r < nrows; r += 2 * step) {
    const bool two = r + step < nrows;
    uint4 q[2][2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      if (e && !two) continue;
      q[e][0] = *reinterpret_cast<const uint4*>(src + (r + e * step) * rp);
      if (!XBF) q[e][1] = *reinterpret_cast<const uint4*>(src + (r + e * step) * rp + 16);
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      if (e && !two) continue;
      const int u = r + e * step;
      uint4 o = chunk8<XBF, BN>(q[e], af, relu);
      if (HALO == 2) {
        const uint4 zero = make_uint4(0, 0, 0, 0);
        const int W = 1 << lgw, H = 1 << ylo, x = u & (W - 1), y = (u >> lgw) & (H - 1);
        const int i0 = u >> (lgw + ylo) << (lgw + ylo);
#pragma unroll 1
        for (int r3 = 0; r3 < 9; r3 += 3) {
          const int dy = y + 1 - r3 / 3;
          const bool in = dy >= 0 && dy < H;
          uint8_t* row = dst + (r3 * pitch << lg) + (i0 + ((dy & (H - 1)) << lgw)) * 16;
#pragma unroll
          for (int s = 0; s < 3; ++s) {
            const int c = x + 1 - s;
            *reinterpret_cast<uint4*>(row + (s * pitch << lg) + (c & (W - 1)) * 16) = in && c >= 0 && c < W ? o : zero;
          }
        }
      } else if (HALO) {
        const uint4 zero = make_uint4(0, 0, 0, 0);
        const int y = u >> lgw, W = 1 << lgw, x = u & (W - 1);
        if (y < ylo || y >= yhi) o = zero;
#pragma unroll
        for (int s = 0; s < 3; ++s) {
          const int c = x + 1 - s;
          *reinterpret_cast<uint4*>(dst + (s * pitch << lg) + (u - x + (c & (W - 1))) * 16) = c >= 0 && c < W ? o : zero;
        }
      } else {
        *reinterpret_cast<uint4*>(dst + u * 16) = o;
      }
    }
  }
}

// ANY: a 3x3 launch with small images or several blocks of output channels;
// without, the code of both folds away
template <int KS, bool ANY>
__device__ __forceinline__ void wg_body(const ConvDesc* __restrict__ tab, const int* __restrict__ ts, int total,
                                        const Rings& rg, int32_t* status) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw0 = smem_u32(smem_raw);
  const uint32_t base = (raw0 + 1023u) & ~1023u;
  uint8_t* const gbase = smem_raw + (base - raw0);
  // [operand ring | raw ring | Shared]: an M side with fewer than 128 channels
  // reads up to kMReach bytes on, into the raw ring at most
  const int off_raw = rg.no * rg.opb;
  Shared& sh = *reinterpret_cast<Shared*>(gbase + rings_bytes(rg));
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kMaxRing; ++s) {
      mbar_init(smem_u32(&sh.raw_full[s]), 1);
      mbar_init(smem_u32(&sh.raw_empty[s]), kT);
      mbar_init(smem_u32(&sh.op_full[s]), kT);
      mbar_init(smem_u32(&sh.op_empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&sh.tfull[b]), 1);
      mbar_init(smem_u32(&sh.tempty[b]), kE);
    }
    mbar_init(smem_u32(&sh.drain), 1);
    sh.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMma) tmem_alloc(smem_u32(&sh.tmem), kTmemCols);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = sh.tmem;
  volatile int* abort_flag = &sh.abort_flag;
  // accumulator buffers: two where every instance of the launch fits (the
  // rule depends on the kernel alone: 1x1 <= 2 x 64 columns, 3x3 <= 9 x 32)
  constexpr int kBufs = KS == 1 ? 2 : 1;
  constexpr int kBufCols = KS == 1 ? 128 : 0;

  if (warp == kProducer) {
    // ================================================= TMA producer
    if (elect_one()) {
      Cursor cr(rg.nr);
      uint32_t n = 0;
      bool ok = true;
      for (Walk w(tab, ts, total); w.more() && ok; w.next(tab, ts)) {
        const ConvDesc* d = w.d;
        const Geo g = geo<KS>(d);
        const int pbeg = w.tm * d->pix_per_split, pend = min(g.rows, pbeg + d->pix_per_split);
        const uint32_t bytes = (uint32_t)(g.p.xrows * g.p.xch * (g.xbf ? 2 : 4) + g.p.kp * g.p.ych * 4);
        const int yb = ANY ? w.tn / wg_xblocks(KS, g.C) : 0, xb = w.tn - (ANY ? yb * wg_xblocks(KS, g.C) : 0);
        const int up = KS == 3 && !(ANY && g.p.small) ? g.W : 0;  // the row above
        for (int p = pbeg; p < pend; p += g.p.kp) {
          if (!mbar_wait(smem_u32(&sh.raw_empty[cr.s]), cr.ph ^ 1, abort_flag)) { ok = false; break; }
          const uint32_t full = smem_u32(&sh.raw_full[cr.s]);
          const uint32_t slot = base + off_raw + cr.s * rg.rawb;
          mbar_expect_tx(full, bytes);
          tma_load_2d(slot, d->tma_a, xb * g.p.xch, p - up, full);
          tma_load_2d(slot + g.p.yoff, d->tma_b, ANY ? yb * g.p.ych : 0, p, full);
          cr.next();
          ++n;
        }
      }
      if (!ok) { sh.abort_flag = 1; atomicExch(status, 3); }
      // the copies of the last slots issued must land before the CTA exits
      for (uint32_t i = n > (uint32_t)rg.nr ? n - rg.nr : 0; i < n; ++i)
        mbar_wait_drain(smem_u32(&sh.raw_full[i % rg.nr]), (i / rg.nr) & 1);
    }
    __syncwarp();
  } else if (warp == kMma) {
    // ================================================= MMA issuer
    if (elect_one()) {
      Cursor co(rg.no), cb(kBufs);
      bool ok = true, issued = false;
      for (Walk w(tab, ts, total); w.more() && ok; w.next(tab, ts)) {
        const ConvDesc* d = w.d;
        const Geo g = geo<KS>(d);
        const int pbeg = w.tm * d->pix_per_split, pend = min(g.rows, pbeg + d->pix_per_split);
        const uint32_t idesc = idesc_bf16(128, (KS == 3 ? 3 : 1) * g.p.nch) | (1u << 15) | (1u << 16);  // both operands MN-major
        const uint32_t tacc = tmem + cb.s * kBufCols;
        if (!mbar_wait(smem_u32(&sh.tempty[cb.s]), cb.ph ^ 1, abort_flag)) { ok = false; break; }
        uint32_t acc = 0;
        for (int p = pbeg; p < pend; p += g.p.kp) {
          if (!mbar_wait(smem_u32(&sh.op_full[co.s]), co.ph, abort_flag)) { ok = false; break; }
          fence_after();
          const uint32_t a_addr = base + co.s * rg.opb, b_addr = a_addr + g.p.boff;
          // (start addresses count 16-byte units: one pixel row)
          const uint64_t ad = nosw_desc(a_addr, 128, g.p.apitch);
          const int steps = g.p.kp >> 4;
          if (KS == 1) {
            const uint64_t bd = nosw_desc(b_addr, 128, g.p.bpitch);
            for (int j = 0; j < steps; ++j) {
              mma_bf16(tacc, ad + j * 16, bd + j * 16, idesc, acc | j ? 1u : 0u);
              // channels 128 .. 255 of the M side
              if (g.p.mch > 128)
                mma_bf16(tacc + 64, ad + (16 * g.p.apitch >> 4) + j * 16, bd + j * 16, idesc, acc | j ? 1u : 0u);
            }
          } else {
            const uint64_t bd = nosw_desc(b_addr, 128, g.p.bpitch);
            const int rs = ANY && g.p.small ? 3 * (g.p.nch >> 3) * (g.p.bpitch >> 4) : g.W;  // between tap rows
            for (int j = 0; j < steps; ++j)
#pragma unroll
              for (int r = 0; r < 3; ++r)
                mma_bf16(tacc + r * 3 * g.p.nch, ad + j * 16, bd + j * 16 + r * rs, idesc, acc | j ? 1u : 0u);
          }
          acc = 1;
          issued = true;
          mma_commit(smem_u32(&sh.op_empty[co.s]));
          co.next();
        }
        if (ok) mma_commit(smem_u32(&sh.tfull[cb.s]));
        cb.next();
      }
      if (!ok) {
        sh.abort_flag = 1;
        atomicExch(status, 3);
        if (issued) {
          mma_commit(smem_u32(&sh.drain));
          mbar_wait_drain(smem_u32(&sh.drain), 0);
        }
      }
    }
    __syncwarp();
  } else if (warp < kE0) {
    // ================================================= transform
    // Warps run independently (each arrives for itself), so a ring of several
    // slots lets them work on different k-steps.
    const int t = threadIdx.x - 32 * kT0;
    Cursor cr(rg.nr), co(rg.no);
    bool ok = true;
    for (Walk w(tab, ts, total); w.more(); w.next(tab, ts)) {
      const ConvDesc* d = w.d;
      const Geo g = geo<KS>(d);
      const int pbeg = w.tm * d->pix_per_split, pend = min(g.rows, pbeg + d->pix_per_split);
      const int relu = g.bn ? d->x.relu : 0;
      const int lgx = 28 - __clz(g.p.xch), lgy = 28 - __clz(ANY ? g.p.ych : g.K);  // log2 of the chunks a pixel
      const int xb = ANY ? w.tn % wg_xblocks(KS, g.C) : w.tn;
      Affine af, none{};
      if (g.bn) af.load(d->x.scale, d->x.shift, xb * g.p.xch + (t & ((1 << lgx) - 1)) * 8);
      // which side x and dY are, their planes in the operand slot
      const int xoff = g.p.x_is_a ? 0 : g.p.boff, yoff = g.p.x_is_a ? g.p.boff : 0;
      const int xpitch = g.p.x_is_a ? g.p.apitch : g.p.bpitch, ypitch = g.p.x_is_a ? g.p.bpitch : g.p.apitch;
      int y0 = KS == 3 ? (pbeg >> g.p.lgw) % g.H : 0;  // first image row of the k-step
      for (int p = pbeg; p < pend; p += g.p.kp, cr.next(), co.next()) {
        if (ok) ok = mbar_wait(smem_u32(&sh.raw_full[cr.s]), cr.ph, abort_flag);
        if (ok) ok = mbar_wait(smem_u32(&sh.op_empty[co.s]), co.ph ^ 1, abort_flag);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) { sh.abort_flag = 1; continue; }
        const uint8_t* raw = gbase + off_raw + cr.s * rg.rawb;
        uint8_t* op = gbase + co.s * rg.opb;
        rows_to_planes<false, false, 0>(raw + g.p.yoff, op + yoff, g.p.kp, lgy, ypitch, t, none, 0, 0, 0, 0);
        const int ylo = y0 == 0 ? 1 : 0, yhi = y0 + g.p.krows == g.H ? g.p.krows + 1 : g.p.krows + 2;
        if (ANY && g.p.small) {
          const int lgh = 31 - __clz(g.H);
          if (g.xbf) {
            if (g.bn) rows_to_planes<true, true, 2>(raw, op + xoff, g.p.xrows, lgx, xpitch, t, af, relu, g.p.lgw, lgh, 0);
            else rows_to_planes<true, false, 2>(raw, op + xoff, g.p.xrows, lgx, xpitch, t, af, 0, g.p.lgw, lgh, 0);
          } else {
            if (g.bn) rows_to_planes<false, true, 2>(raw, op + xoff, g.p.xrows, lgx, xpitch, t, af, relu, g.p.lgw, lgh, 0);
            else rows_to_planes<false, false, 2>(raw, op + xoff, g.p.xrows, lgx, xpitch, t, af, 0, g.p.lgw, lgh, 0);
          }
        } else if (g.xbf) {
          if (g.bn)
            rows_to_planes<true, true, KS == 3>(raw, op + xoff, g.p.xrows, lgx, xpitch, t, af, relu, g.p.lgw, ylo, yhi);
          else
            rows_to_planes<true, false, KS == 3>(raw, op + xoff, g.p.xrows, lgx, xpitch, t, af, 0, g.p.lgw, ylo, yhi);
        } else {
          if (g.bn)
            rows_to_planes<false, true, KS == 3>(raw, op + xoff, g.p.xrows, lgx, xpitch, t, af, relu, g.p.lgw, ylo, yhi);
          else
            rows_to_planes<false, false, KS == 3>(raw, op + xoff, g.p.xrows, lgx, xpitch, t, af, 0, g.p.lgw, ylo, yhi);
        }
        if (KS == 3) {
          y0 += g.p.krows;
          if (y0 >= g.H) y0 = 0;
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(smem_u32(&sh.raw_empty[cr.s]));
          mbar_arrive(smem_u32(&sh.op_full[co.s]));
        }
      }
    }
    if (!ok) { sh.abort_flag = 1; atomicExch(status, 3); }
  } else {
    // ================================================= epilogue
    const int q = warp & 3;
    Cursor cb(kBufs);
    bool ok = true;
    for (Walk w(tab, ts, total); w.more(); w.next(tab, ts), cb.next()) {
      const ConvDesc* d = w.d;
      const Geo g = geo<KS>(d);
      if (ok) ok = mbar_wait(smem_u32(&sh.tfull[cb.s]), cb.ph, abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) { sh.abort_flag = 1; continue; }
      fence_after();
      const uint32_t tacc = tmem + cb.s * kBufCols + ((uint32_t)(q * 32) << 16);
      // blocks of 16 accumulator columns: 1x1 (M half, N) rows of nch floats;
      // 3x3 (tap, N) rows of 9 C floats
      const int per = g.p.nch >> 4;
      const int yb = ANY ? w.tn / wg_xblocks(KS, g.C) : 0, xb = w.tn - (ANY ? yb * wg_xblocks(KS, g.C) : 0);
      const int blocks = (KS == 1 ? (g.p.mch > 128 ? 2 : 1) : 9) * per;
      for (int b = 0; b < blocks; ++b) {
        const int outer = b / per, n = (b - outer * per) * 16;
        const int m = q * 32 + lane + (KS == 1 ? outer * 128 : 0);
        if (q * 32 + (KS == 1 ? outer * 128 : 0) >= g.p.mch) continue;  // (the whole warp)
        uint32_t a[16];
        tmem_ld16_nowait(tacc + outer * (KS == 1 ? 64 : g.p.nch) + n, a);
        tmem_wait_ld(a);
        if (m < g.p.mch) {
          float* out = KS == 1 ? d->dw_part + ((int64_t)w.tm * g.p.mch + m) * g.p.nch + n
                               : d->dw_part + (((int64_t)w.tm * g.K + yb * 128 + m) * 9 + outer) * g.C + xb * g.p.nch + n;
#pragma unroll
          for (int i = 0; i < 4; ++i)
            reinterpret_cast<uint4*>(out)[i] = make_uint4(a[4 * i], a[4 * i + 1], a[4 * i + 2], a[4 * i + 3]);
        }
      }
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&sh.tempty[cb.s]));
    }
    if (!ok) { sh.abort_flag = 1; atomicExch(status, 3); }
  }
  fence_before();
  __syncthreads();
  if (warp == kMma) {
    fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

__global__ void __launch_bounds__(kThreads, 1) k_wg_pw(const ConvDesc* __restrict__ tab, const int* __restrict__ ts,
                                                       int total, const Rings rg, int32_t* status) {
  wg_body<1, false>(tab, ts, total, rg, status);
}
template <bool ANY>
__global__ void __launch_bounds__(kThreads, 1) k_wg_3x3(const ConvDesc* __restrict__ tab, const int* __restrict__ ts,
                                                        int total, const Rings rg, int32_t* status) {
  wg_body<3, ANY>(tab, ts, total, rg, status);
}

}  // namespace

bool wg_fits(int raw_bytes, int op_bytes) {
  Rings r;
  return plan_rings(raw_bytes, op_bytes, r);
}

cudaError_t launch_conv_wg(int ksize, int any, const ConvDesc* tab, const int* ts, int total, int raw_bytes, int op_bytes,
                           int32_t* status, cudaStream_t st, int max_ctas) {
  if (total <= 0) return cudaSuccess;
  Rings r;
  if (raw_bytes <= 0 || op_bytes <= 0 || (raw_bytes & 1023) || (op_bytes & 1023) || !plan_rings(raw_bytes, op_bytes, r))
    return cudaErrorInvalidValue;
  auto kern = ksize != 3 ? k_wg_pw : any ? k_wg_3x3<true> : k_wg_3x3<false>;
  cudaError_t e = set_smem_attr_once(ksize != 3 ? 15 : any ? 21 : 16, reinterpret_cast<const void*>(kern), kSmemBudget);
  if (e != cudaSuccess) return e;
  const int sms = device_sm_count();
  int grid = total < sms ? total : sms;
  if (max_ctas > 0 && grid > max_ctas) grid = max_ctas;
  kern<<<grid, kThreads, kFixed + rings_bytes(r), st>>>(tab, ts, total, r, status);
  return cudaGetLastError();
}

}  // namespace pnn
