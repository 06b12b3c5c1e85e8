// Grouped 3x3 stride-1 convolutions of the bottleneck stacks with at most 64
// channels, forward and data gradient, on the 5th-generation tensor cores: the
// 3x3 counterpart of k_pw_conv.cu (same roles, same epilogue).
//
// A tile is a patch of 8 x 16 pixels of one image, or two whole 8 x 8 images.
// Its M rows run patch row by patch row, so each 8-row core matrix of the A
// operand is one row segment and the segments are a fixed distance apart in the
// halo around the patch; tap (r, s) is then the same halo read from another
// start (a descriptor offset: no-swizzle operands start at any 16-byte row).
// Every input pixel is transformed and stored once -- the former kernel stored
// three column-shifted copies of a full-width halo, which with the padding
// logic was 54 % of its time -- and the hardware's zero fill of a 4-D box brings
// the image border.  (8 x 8 images cannot share a halo at a uniform distance;
// theirs is stored in three row-shifted copies.)  A k-step is 16 channels: two
// planes of 16-byte pixels, and the nine taps' weights of those channels in the
// operand's own layout (k_wtrans packs them after every update), so that one
// contiguous copy brings them: as 18 boxes of 16-byte rows they cost the
// producer 200 cycles each and bounded the kernel.
// Grouped launches of the 8-subnetwork ResNet-1001 (batch 256, 64 px), kernels of
// k_tc_conv.cu -> now: forward 160 -> 62 us, data gradient (+ BN-backward sums)
// 133 -> 90 us; bound by per-tile latencies (a tile is 128 x 16 outputs).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "narrow_epilogue.cuh"
#include "pnn.h"
#include "pnn_internal.h"
#include "tc_pair.cuh"
#include "tc_ptx.cuh"

namespace pnn {
namespace {

using namespace tc;

constexpr int kT = 6, kE = 8;
constexpr int kProducer = 0, kMma = 1, kT0 = 2, kE0 = kT0 + kT;
constexpr int kThreads = 32 * (2 + kT + kE);
constexpr int kNT = 32 * kT;
constexpr int kGroups = kE / 4;
constexpr int kMaxRing = 4;
constexpr int kAcc = 4, kAccCols = 64;
constexpr int kSmemBudget = 227 * 1024;
static_assert(kE0 % 4 == 0, "epilogue groups start at a TMEM lane quarter");

struct Shared {
  uint64_t raw_full[kMaxRing], raw_empty[kMaxRing];
  uint64_t op_full[kMaxRing], op_empty[kMaxRing];
  uint64_t u_full[kMaxRing], u_empty[kMaxRing];
  uint64_t tfull[kAcc], tempty[kAcc];
  uint64_t drain;
  uint32_t tmem;
  int abort_flag;
};

struct Rings {
  int nr, no, nu, rawb, opb, wb, ub;
};
__host__ __device__ inline int rings_bytes(const Rings& r) { return r.nr * r.rawb + r.no * r.opb + r.nu * r.ub; }
template <int MODE>
constexpr int fixed_bytes() {
  return 1024 + (int)sizeof(Shared) + kE * stage_bytes(MODE) + kGroups * kRedBytes;
}
template <int MODE>
bool plan_rings(const C3Slots& s, Rings& r) {
  r = Rings{2, 2, 2, s.raw, s.op, s.wt, s.wt + s.x};
  const int avail = kSmemBudget - fixed_bytes<MODE>();
  if (rings_bytes(r) > avail) return false;
  for (int* n : {&r.nr, &r.no, &r.nu, &r.nr, &r.no, &r.nu}) {
    if (*n >= kMaxRing) continue;
    ++*n;
    if (rings_bytes(r) > avail) --*n;
  }
  return true;
}

struct Geo {
  int rows, n, nk, H, W, tx, tpi;  // GEMM M and N; 16-channel k-steps; patches a row and an image
  bool whole;                      // two whole 8 x 8 images
};
template <int MODE>
__device__ __forceinline__ Geo geo(const ConvDesc* d) {
  Geo g;
  g.H = d->H;
  g.W = d->W;
  g.rows = d->B * d->H * d->W;
  g.n = MODE == FWD ? d->K : d->C;
  g.nk = (MODE == FWD ? d->C : d->K) >> 4;
  g.whole = c3_whole(d->H, d->W);
  g.tx = d->W >> 3;
  g.tpi = g.tx * (d->H >> 4);
  return g;
}
// the patch of a tile
struct Patch {
  int img, y0, x0;
};
__device__ __forceinline__ Patch patch(const Geo& g, int tm) {
  Patch p;
  if (g.whole) {
    p.img = 2 * tm;
    p.y0 = p.x0 = 0;
  } else {
    p.img = tm / g.tpi;
    const int r = tm - p.img * g.tpi, ty = r / g.tx;
    p.y0 = ty * 16;
    p.x0 = (r - ty * g.tx) * 8;
  }
  return p;
}
// where a warp's 32 rows of the output tile go: four rows of 8 pixels
struct PatchDst {
  Patch p;
  bool whole;
  __device__ __forceinline__ void put(const void* map, int n, int q, uint32_t src, bool add) const {
    const int y = whole ? (q & 1) * 4 : p.y0 + 4 * q, img = whole ? p.img + (q >> 1) : p.img;
    if (add) tma_reduce_add_4d(map, n, p.x0, y, img, src);
    else tma_store_4d(map, n, p.x0, y, img, src);
  }
};

// ------------------------------------------------------------ transform
// Raw pixels of one k-step ([pixels][16 channels], dense) -> two planes of 8
// channels.  Thread t takes chunk t & 1 of pixels t / 2, + 96, ...
template <bool XBF, bool BN>
__device__ __forceinline__ void transform_px(const uint8_t* __restrict__ raw, uint8_t* __restrict__ op, int t,
                                             const uint64_t (&sc)[4], const uint64_t (&sf)[4], int relu, const Geo& g,
                                             const Patch& pt) {
  const int cc = t & 1;
  const uint8_t* src = raw + cc * (XBF ? 16 : 32);
  uint8_t* dst = op + cc * c3_plane(g.whole);
  const int npx = g.whole ? 128 : 180;
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int u = (t >> 1) + e * (kNT / 2);
    if (u >= npx) break;
    uint4 q0 = *reinterpret_cast<const uint4*>(src + u * (XBF ? 32 : 64)), q1 = make_uint4(0, 0, 0, 0);
    if (!XBF) q1 = *reinterpret_cast<const uint4*>(src + u * 64 + 16);
    uint32_t o[4];
    if (XBF) {
      const uint32_t w[4] = {q0.x, q0.y, q0.z, q0.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        o[i] = BN ? pack2(fma2(sc[i], bf2(w[i]), sf[i])) : w[i];
        if (BN && relu) o[i] = relu2(o[i]);
      }
    } else {
      const uint32_t w[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint64_t v = pk2(__uint_as_float(w[2 * i]), __uint_as_float(w[2 * i + 1]));
        o[i] = BN ? pack2(fma2(sc[i], v, sf[i])) : pack2(v);
        if (BN && relu) o[i] = relu2(o[i]);
      }
    }
    const uint4 zero = make_uint4(0, 0, 0, 0);
    uint4 v = make_uint4(o[0], o[1], o[2], o[3]);
    if (!g.whole) {
      // halo row and column of the pixel; outside the image the value is zero, not BN(0)
      const int hy = u / 10, hx = u - 10 * hy;
      const int y = pt.y0 - 1 + hy, x = pt.x0 - 1 + hx;
      if (y < 0 || y >= g.H || x < 0 || x >= g.W) v = zero;
      *reinterpret_cast<uint4*>(dst + u * 16) = v;
    } else {
      // copy r holds image row y + r - 1 at row y (of 8 a image): this pixel goes to rows y + 1, y, y - 1;
      // the row that falls out of the image is the one the copy needs zero
      const int x = u & 7, y = (u >> 3) & 7, i8 = (u >> 6) * 8;
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        const int row = (y + 1 - r) & 7;
        const bool in = y + 1 - r >= 0 && y + 1 - r < 8;
        *reinterpret_cast<uint4*>(dst + (r * 160 + (i8 + row) * 10 + x + 1) * 16) = in ? v : zero;
      }
    }
  }
  if (g.whole) {
    // the zero columns: 3 copies x 16 rows x 2
    const int e = t >> 1;  // 0 .. 95
    *reinterpret_cast<uint4*>(dst + ((e >> 5) * 160 + ((e >> 1) & 15) * 10 + (e & 1) * 9) * 16) = make_uint4(0, 0, 0, 0);
  }
}

template <int MODE>
__device__ __forceinline__ void c3_body(const ConvDesc* __restrict__ tab, const int* __restrict__ ts, int ninst,
                                        int total, const Rings& rg, int32_t* status) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw0 = smem_u32(smem_raw);
  const uint32_t base = (raw0 + 1023u) & ~1023u;
  uint8_t* const gbase = smem_raw + (base - raw0);
  // [unit ring | output staging | reduction | operand ring | raw ring | Shared]
  // (the swizzled tiles first: every size before them is a multiple of 1024)
  uint8_t* const stage0 = gbase + rg.nu * rg.ub;
  uint8_t* const red0 = stage0 + kE * stage_bytes(MODE);
  const int off_op = rg.nu * rg.ub + kE * stage_bytes(MODE) + kGroups * kRedBytes;
  const int off_raw = off_op + rg.no * rg.opb;
  Shared& sh = *reinterpret_cast<Shared*>(gbase + off_raw + rg.nr * rg.rawb);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kMaxRing; ++s) {
      mbar_init(smem_u32(&sh.raw_full[s]), 1);
      mbar_init(smem_u32(&sh.raw_empty[s]), kT);
      mbar_init(smem_u32(&sh.op_full[s]), kT);
      mbar_init(smem_u32(&sh.op_empty[s]), 1);
      mbar_init(smem_u32(&sh.u_full[s]), 1);
      // the MMA's commit and the readers of X: the tile's four epilogue warps, or (no X) the MMA thread for them
      mbar_init(smem_u32(&sh.u_empty[s]), 1 + 4);
    }
    for (int b = 0; b < kAcc; ++b) {
      mbar_init(smem_u32(&sh.tfull[b]), 1);
      mbar_init(smem_u32(&sh.tempty[b]), 4);
    }
    mbar_init(smem_u32(&sh.drain), 1);
    sh.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMma) tmem_alloc(smem_u32(&sh.tmem), kAcc * kAccCols);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = sh.tmem;
  volatile int* abort_flag = &sh.abort_flag;

  if (warp == kProducer) {
    // ================================================= TMA producer
    if (elect_one()) {
      Cursor cr(rg.nr), cu(rg.nu);
      uint32_t ka = 0, u = 0;  // raw and unit slots issued
      bool ok = true;
      Geo g{};
      const void *ma = nullptr, *mx = nullptr;
      const uint8_t* wt = nullptr;
      uint32_t abytes = 0;
      int off = 0;
      for (Walk w(tab, ts, ninst, total); w.more() && ok; w.next(tab, ts)) {
        if (w.fresh) {
          const ConvDesc* d = w.d;
          g = geo<MODE>(d);
          ma = d->tma_a;
          mx = has_x<MODE>(d) ? d->tma_x : nullptr;
          wt = static_cast<const uint8_t*>(d->w);
          abytes = (uint32_t)(c3_raw_px(g.whole) * 16 * (MODE == FWD && d->x.dt == DT_BF16 ? 2 : 4));
          off = g.whole ? 0 : 1;
          tma_prefetch_map(ma);
          if (mx) tma_prefetch_map(mx);
        }
        const Patch p = patch(g, w.tm);
        const uint32_t wbytes = (uint32_t)c3_wt_bytes(g.n);
        for (int kt = 0; kt < g.nk; ++kt) {
          if (!mbar_wait(smem_u32(&sh.raw_empty[cr.s]), cr.ph ^ 1, abort_flag)) { ok = false; break; }
          const uint32_t full = smem_u32(&sh.raw_full[cr.s]);
          mbar_expect_tx(full, abytes);
          tma_load_4d(base + off_raw + cr.s * rg.rawb, ma, kt * 16, p.x0 - off, p.y0 - off, p.img, full);
          cr.next();
          ++ka;
          if (!mbar_wait(smem_u32(&sh.u_empty[cu.s]), cu.ph ^ 1, abort_flag)) { ok = false; break; }
          const uint32_t uf = smem_u32(&sh.u_full[cu.s]);
          const uint32_t slot = base + cu.s * rg.ub;
          const bool x = mx != nullptr && kt == g.nk - 1;
          mbar_expect_tx(uf, wbytes + (x ? (uint32_t)(kTcBM * g.n * 2) : 0u));
          bulk_load(slot, wt + (size_t)kt * wbytes, wbytes, uf);
          if (x) tma_load_4d(slot + rg.wb, mx, 0, p.x0, p.y0, p.img, uf);
          cu.next();
          ++u;
        }
      }
      if (!ok) { sh.abort_flag = 1; atomicExch(status, 3); }
      // the copies of the last slots issued must land before the CTA exits
      for (uint32_t i = ka > (uint32_t)rg.nr ? ka - rg.nr : 0; i < ka; ++i)
        mbar_wait_drain(smem_u32(&sh.raw_full[i % rg.nr]), (i / rg.nr) & 1);
      for (uint32_t i = u > (uint32_t)rg.nu ? u - rg.nu : 0; i < u; ++i)
        mbar_wait_drain(smem_u32(&sh.u_full[i % rg.nu]), (i / rg.nu) & 1);
    }
    __syncwarp();
  } else if (warp == kMma) {
    // ================================================= MMA issuer
    if (elect_one()) {
      Cursor co(rg.no), cu(rg.nu), cb(kAcc);
      bool ok = true, issued = false;
      Geo g{};
      bool hx = false;
      uint32_t idesc = 0;
      int rs = 0;  // pixels between the starts of tap rows
      for (Walk w(tab, ts, ninst, total); w.more() && ok; w.next(tab, ts), cb.next()) {
        if (w.fresh) {
          g = geo<MODE>(w.d);
          hx = has_x<MODE>(w.d);
          idesc = idesc_bf16(kTcBM, g.n);
          rs = g.whole ? 160 : 10;
        }
        const uint32_t tacc = tmem + cb.s * kAccCols;
        if (!mbar_wait(smem_u32(&sh.tempty[cb.s]), cb.ph ^ 1, abort_flag)) { ok = false; break; }
        for (int kt = 0; kt < g.nk; ++kt) {
          if (!mbar_wait(smem_u32(&sh.u_full[cu.s]), cu.ph, abort_flag)) { ok = false; break; }
          if (!mbar_wait(smem_u32(&sh.op_full[co.s]), co.ph, abort_flag)) { ok = false; break; }
          fence_after();
          // (descriptor starts count 16-byte units: one pixel, one weight row)
          const uint64_t ad = nosw_desc(base + off_op + co.s * rg.opb, c3_plane(g.whole), 160);
          const uint64_t bd = nosw_desc(base + cu.s * rg.ub, 9 * g.n * 16, 128);
#pragma unroll
          for (int tap = 0; tap < 9; ++tap) {
            const int r = MODE == FWD ? tap / 3 : 2 - tap / 3, s = MODE == FWD ? tap % 3 : 2 - tap % 3;
            mma_bf16(tacc, ad + r * rs + s, bd + tap * g.n, idesc, (kt | tap) ? 1u : 0u);
          }
          issued = true;
          if (!(hx && kt == g.nk - 1)) mbar_arrive_n(smem_u32(&sh.u_empty[cu.s]), 4);
          mma_commit(smem_u32(&sh.u_empty[cu.s]));
          mma_commit(smem_u32(&sh.op_empty[co.s]));
          co.next();
          cu.next();
        }
        if (ok) mma_commit(smem_u32(&sh.tfull[cb.s]));
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
    // (warps run independently; one whose wait fails stops working but keeps walking)
    const int t = threadIdx.x - 32 * kT0;
    Cursor cr(rg.nr), co(rg.no);
    bool ok = true;
    uint64_t sc[4] = {}, sf[4] = {};
    Geo g{};
    bool bn = false, xbf = false;
    int relu = 0;
    for (Walk w(tab, ts, ninst, total); w.more(); w.next(tab, ts)) {
      const ConvDesc* d = w.d;
      if (w.fresh) {
        g = geo<MODE>(d);
        bn = MODE == FWD && d->x.scale != nullptr;
        xbf = MODE == FWD && d->x.dt == DT_BF16;
        relu = bn ? d->x.relu : 0;
      }
      const Patch p = patch(g, w.tm);
      for (int kt = 0; kt < g.nk; ++kt, cr.next(), co.next()) {
        if (bn && (w.fresh || g.nk > 1)) {
          // this thread's 8 channels; one k-step keeps them until the instance changes
          const int c = kt * 16 + (t & 1) * 8;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float2 a = __ldg(reinterpret_cast<const float2*>(d->x.scale + c) + i);
            const float2 b = __ldg(reinterpret_cast<const float2*>(d->x.shift + c) + i);
            sc[i] = pk2(a.x, a.y);
            sf[i] = pk2(b.x, b.y);
          }
        }
        if (ok) ok = mbar_wait(smem_u32(&sh.raw_full[cr.s]), cr.ph, abort_flag);
        if (ok) ok = mbar_wait(smem_u32(&sh.op_empty[co.s]), co.ph ^ 1, abort_flag);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) { sh.abort_flag = 1; continue; }
        const uint8_t* raw = gbase + off_raw + cr.s * rg.rawb;
        uint8_t* op = gbase + off_op + co.s * rg.opb;
        if (MODE == DGRAD) {
          transform_px<false, false>(raw, op, t, sc, sf, 0, g, p);
        } else if (xbf) {
          if (bn) transform_px<true, true>(raw, op, t, sc, sf, relu, g, p);
          else transform_px<true, false>(raw, op, t, sc, sf, 0, g, p);
        } else {
          if (bn) transform_px<false, true>(raw, op, t, sc, sf, relu, g, p);
          else transform_px<false, false>(raw, op, t, sc, sf, 0, g, p);
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
    const int ew = warp - kE0, q = warp & 3, eg = ew >> 2;
    uint8_t* const st = stage0 + ew * stage_bytes(MODE);
    EpiState es{reinterpret_cast<float2*>(red0 + eg * kRedBytes), 0, 2 + eg};
    Cursor cu(rg.nu), cb(kAcc);
    int turn = 0, sbuf = 0;
    const bool leader = elect_one();  // issues and waits for this warp's stores
    bool ok = true;
    Geo g{};
    EpiArgs ea{};
    for (Walk w(tab, ts, ninst, total); w.more(); w.next(tab, ts)) {
      if (w.fresh) {
        g = geo<MODE>(w.d);
        ea.load<MODE>(w.d);
      }
      // the tile's last k-step holds X
      for (int i = 1; i < g.nk; ++i) cu.next();
      const int us = cu.s, b = cb.s;
      const uint32_t uph = cu.ph, bph = cb.ph;
      cu.next();
      cb.next();
      const bool mine = turn == eg;
      if (++turn == kGroups) turn = 0;
      if (!mine) continue;
      const int m0 = w.tm * kTcBM;
      if (ok) ok = mbar_wait(smem_u32(&sh.tfull[b]), bph, abort_flag);
      if (ok && ea.hx) ok = mbar_wait(smem_u32(&sh.u_full[us]), uph, abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      float2* redw = es.red + es.rbuf * 256 + q * 64;
      if (ok) {
        fence_after();
        const uint32_t tacc = tmem + b * kAccCols + ((uint32_t)(q * 32) << 16);
        const uint8_t* x = gbase + us * rg.ub + rg.wb;
        const uint32_t te = smem_u32(&sh.tempty[b]), ue = smem_u32(&sh.u_empty[us]);
        const PatchDst dst{patch(g, w.tm), g.whole};
        if (MODE == FWD) {
          if (g.n == 64) unit_fwd<64>(ea, dst, tacc, q, lane, g.rows, m0, 0, x, st, redw, te, ue, leader);
          else if (g.n == 32) unit_fwd<32>(ea, dst, tacc, q, lane, g.rows, m0, 0, x, st, redw, te, ue, leader);
          else unit_fwd<16>(ea, dst, tacc, q, lane, g.rows, m0, 0, x, st, redw, te, ue, leader);
        } else {
          if (g.n == 64) unit_dgrad<64>(ea, dst, tacc, q, lane, g.rows, m0, 0, x, st, sbuf, redw, te, ue, leader);
          else if (g.n == 32) unit_dgrad<32>(ea, dst, tacc, q, lane, g.rows, m0, 0, x, st, sbuf, redw, te, ue, leader);
          else unit_dgrad<16>(ea, dst, tacc, q, lane, g.rows, m0, 0, x, st, sbuf, redw, te, ue, leader);
        }
      } else {
        sh.abort_flag = 1;
      }
      if (ea.stats) {
        float* p = ea.part + (int64_t)w.tm * g.n * 2;
        if (g.n == 64) merge_partials<MODE, 64>(es, ok, q, lane, g.rows, m0, p);
        else if (g.n == 32) merge_partials<MODE, 32>(es, ok, q, lane, g.rows, m0, p);
        else merge_partials<MODE, 16>(es, ok, q, lane, g.rows, m0, p);
      }
    }
    // the output stores must complete before the CTA exits
    if (leader) bulk_wait_all();
    __syncwarp();
    if (!ok) { sh.abort_flag = 1; atomicExch(status, 3); }
  }
  fence_before();
  __syncthreads();
  if (warp == kMma) {
    fence_after();
    tmem_dealloc(tmem, kAcc * kAccCols);
  }
}

__global__ void __launch_bounds__(kThreads, 1) k_c3_fwd(const ConvDesc* __restrict__ tab, const int* __restrict__ ts,
                                                        int ninst, int total, const Rings rg, int32_t* status) {
  c3_body<FWD>(tab, ts, ninst, total, rg, status);
}
__global__ void __launch_bounds__(kThreads, 1) k_c3_dgrad(const ConvDesc* __restrict__ tab, const int* __restrict__ ts,
                                                          int ninst, int total, const Rings rg, int32_t* status) {
  c3_body<DGRAD>(tab, ts, ninst, total, rg, status);
}

}  // namespace

cudaError_t launch_conv_c3(int mode, const ConvDesc* tab, const int* ts, int n, int total, const C3Slots& s,
                           int32_t* status, cudaStream_t st, int max_ctas) {
  if (total <= 0) return cudaSuccess;
  if ((s.raw & 127) || (s.op & 127) || (s.wt & 1023) || (s.x & 1023) || s.raw <= 0 || s.op <= 0 || s.wt <= 0)
    return cudaErrorInvalidValue;
  Rings r;
  if (!(mode == FWD ? plan_rings<FWD>(s, r) : plan_rings<DGRAD>(s, r))) return cudaErrorInvalidValue;
  auto kern = mode == FWD ? k_c3_fwd : k_c3_dgrad;
  cudaError_t e = set_smem_attr_once(mode == FWD ? 17 : 18, reinterpret_cast<const void*>(kern), kSmemBudget);
  if (e != cudaSuccess) return e;
  const int sms = device_sm_count();
  int grid = total < sms ? total : sms;
  if (max_ctas > 0 && grid > max_ctas) grid = max_ctas;
  const int smem = (mode == FWD ? fixed_bytes<FWD>() : fixed_bytes<DGRAD>()) + rings_bytes(r);
  kern<<<grid, kThreads, smem, st>>>(tab, ts, n, total, r, status);
  return cudaGetLastError();
}

}  // namespace pnn
