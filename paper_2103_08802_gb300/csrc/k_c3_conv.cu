// Grouped 3x3 stride-1 convolutions, forward and data gradient, on the
// 5th-generation tensor cores: the 3x3 counterpart of k_pw_conv.cu (same roles,
// same epilogue).
//
// A tile is a patch of 8 x 16 pixels of one image, two whole 8 x 8 images, or
// 128 / (H W) smaller ones, by a block of at most 64 output columns.
// Its M rows run patch row by patch row, so each 8-row core matrix of the A
// operand is one row segment and the segments are a fixed distance apart in the
// halo around the patch; tap (r, s) is then the same halo read from another
// start (a descriptor offset: no-swizzle operands start at any 16-byte row).
// Every input pixel is transformed and stored once -- the former kernel stored
// three column-shifted copies of a full-width halo, which with the padding
// logic was 54 % of its time -- and the hardware's zero fill of a 4-D box brings
// the image border.  (8 x 8 images cannot share a halo at a uniform distance;
// theirs is stored in three row-shifted copies, and smaller images in nine, one
// a tap.)  A k-step is 16 channels: two
// planes of 16-byte pixels, and the nine taps' weights of those channels in the
// operand's own layout (k_wtrans packs them after every update), so that one
// contiguous copy brings them: as 18 boxes of 16-byte rows they cost the
// producer 200 cycles each and bounded the kernel.
// Grouped launches of the 8-subnetwork ResNet-1001 (batch 256, 64 px), kernels of
// k_tc_conv.cu -> now: forward 160 -> 58 us, data gradient (+ BN-backward sums)
// 133 -> 74 us; bound by per-tile latencies (a tile is 128 x 16 outputs).  VGG-16
// (batch 128), kernels of k_tc_conv.cu -> now: 128 -> 128 channels at 16 x 16, 4
// instances, forward 204 -> 70 us, data gradient 152 -> 74; 256 -> 256 at 8 x 8, 3
// instances, 171 -> 54 and 120 -> 55; 512 -> 512 at 2 x 2, 116 -> 29 and 80 -> 27.
// Those are 9 MMAs a k-step of N = 64 (about 300 cycles: the read of the M side)
// beside a transform of 400 - 500 by six warps.
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
constexpr int kMaxRing = 4, kMaxX = 8;
constexpr int kAcc = 4, kAccCols = 64;
constexpr int kSmemBudget = 227 * 1024;
static_assert(kE0 % 4 == 0, "epilogue groups start at a TMEM lane quarter");

struct Shared {
  uint64_t raw_full[kMaxRing], raw_empty[kMaxRing];
  uint64_t op_full[kMaxRing], op_empty[kMaxRing];
  uint64_t u_full[kMaxRing], u_empty[kMaxRing];
  uint64_t x_full[kMaxX], x_empty[kMaxX];
  uint64_t tfull[kAcc], tempty[kAcc];
  uint64_t drain;
  uint32_t tmem;
  int abort_flag;
};

// raw pixels, operands, weights of a k-step, second operand of a tile
struct Rings {
  int nr, no, nu, nx, rawb, opb, wb, xb;
};
__host__ __device__ inline int rings_bytes(const Rings& r) {
  return r.nr * r.rawb + r.no * r.opb + r.nu * r.wb + r.nx * r.xb;
}
template <int MODE>
constexpr int fixed_bytes() {
  return 1024 + (int)sizeof(Shared) + kE * stage_bytes(MODE) + kGroups * kRedBytes;
}
template <int MODE>
bool plan_rings(const C3Slots& s, Rings& r) {
  r = Rings{2, 2, 2, s.x > 0, s.raw, s.op, s.wt, s.x};
  const int avail = kSmemBudget - fixed_bytes<MODE>();
  if (rings_bytes(r) > avail) return false;
  // deeper while there is room: X first up to the accumulators in flight
  for (int* n : {&r.nx, &r.nr, &r.no, &r.nu, &r.nx, &r.nr, &r.no, &r.nu, &r.nx, &r.nx, &r.nx, &r.nx}) {
    if (n == &r.nx && !s.x) continue;
    ++*n;
    if (rings_bytes(r) > avail) --*n;
  }
  return true;
}

// two slots of each ring and one second operand fit for the largest instances of c3_ok
// together (fp32 patches, small images, 64 columns), so the launch of a planned group
// cannot fail
template <int MODE>
constexpr bool fits() {
  return fixed_bytes<MODE>() + 2 * (c3_raw_px(C3_PATCH) * 16 * 4 + 2 * c3_plane(C3_SMALL) + c3_wt_bytes(64)) +
             kTcBM * 64 * 2 <= kSmemBudget;
}
static_assert(fits<FWD>() && fits<DGRAD>(), "two slots of each ring");

struct Geo {
  int rows, n, nt, nk, H, W, tx, tpi;  // GEMM M, columns of a block and in all; 16-channel k-steps; patches a row and an image
  int kind, lw, li;                    // C3_PATCH, C3_WHOLE or C3_SMALL; log2 W, log2 H W (whole images)
};
// ANY: a launch with small images or several column blocks; without, the code of both folds away
template <int MODE, bool ANY>
__device__ __forceinline__ Geo geo(const ConvDesc* d) {
  Geo g;
  g.H = d->H;
  g.W = d->W;
  g.rows = d->B * d->H * d->W;
  g.nt = MODE == FWD ? d->K : d->C;
  g.n = ANY ? c3_block(g.nt) : g.nt;
  g.nk = (MODE == FWD ? d->C : d->K) >> 4;
  g.kind = ANY ? c3_kind(d->H, d->W) : (d->H == 8 && d->W == 8 ? C3_WHOLE : C3_PATCH);
  g.lw = 31 - __clz(d->W);
  g.li = ANY ? 31 - __clz(d->H * d->W) : 6;
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
  if (g.kind != C3_PATCH) {
    p.img = tm << (7 - g.li);
    p.y0 = p.x0 = 0;
  } else {
    p.img = tm / g.tpi;
    const int r = tm - p.img * g.tpi, ty = r / g.tx;
    p.y0 = ty * 16;
    p.x0 = (r - ty * g.tx) * 8;
  }
  return p;
}
// where a warp's 32 rows of the output tile go: four rows of 8 pixels, or whole images
template <bool ANY>
struct PatchDst {
  Patch p;
  int kind, li;
  __device__ __forceinline__ void put(const void* map, int n, int q, uint32_t src, bool add) const {
    const int y = kind == C3_WHOLE ? (q & 1) * 4 : !ANY || kind == C3_PATCH ? p.y0 + 4 * q : 0;
    const int img = p.img + (kind == C3_WHOLE ? q >> 1 : !ANY || kind == C3_PATCH ? 0 : q << (5 - li));
    if (add) tma_reduce_add_4d(map, n, p.x0, y, img, src);
    else tma_store_4d(map, n, p.x0, y, img, src);
  }
};

// ------------------------------------------------------------ transform
// Raw pixels of one k-step ([pixels][16 channels], dense) -> two planes of 8
// channels.  Thread t takes chunk t & 1 of pixels t / 2, + 96, ...
// (KIND 0: C3_PATCH or C3_WHOLE, told apart at run time)
template <bool XBF, bool BN, int KIND>
__device__ __forceinline__ void transform_px(const uint8_t* __restrict__ raw, uint8_t* __restrict__ op, int t,
                                             const uint64_t (&sc)[4], const uint64_t (&sf)[4], int relu, const Geo& g,
                                             const Patch& pt) {
  const int kind = KIND ? KIND : g.kind;
  const int cc = t & 1;
  const uint8_t* src = raw + cc * (XBF ? 16 : 32);
  uint8_t* dst = op + cc * c3_plane(kind);
  const int npx = c3_raw_px(kind);
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
    if (kind == C3_PATCH) {
      // halo row and column of the pixel; outside the image the value is zero, not BN(0)
      const int hy = u / 10, hx = u - 10 * hy;
      const int y = pt.y0 - 1 + hy, x = pt.x0 - 1 + hx;
      if (y < 0 || y >= g.H || x < 0 || x >= g.W) v = zero;
      *reinterpret_cast<uint4*>(dst + u * 16) = v;
    } else if (KIND == C3_SMALL) {
      // copy (r, s) holds image pixel (y + r - 1, x + s - 1) at (y, x): this pixel goes to nine places, and
      // where one falls out of the image its wrapped place is the one that the copy needs zero
      const int x = u & (g.W - 1), y = (u >> g.lw) & (g.H - 1), i0 = u >> g.li << g.li;
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        const int dy = y + 1 - r, row = i0 + ((dy & (g.H - 1)) << g.lw);
        const bool in = dy >= 0 && dy < g.H;
#pragma unroll
        for (int s = 0; s < 3; ++s) {
          const int dx = x + 1 - s;
          *reinterpret_cast<uint4*>(dst + ((3 * r + s) * 128 + row + (dx & (g.W - 1))) * 16) =
              in && dx >= 0 && dx < g.W ? v : zero;
        }
      }
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
  if (kind == C3_WHOLE) {
    // the zero columns: 3 copies x 16 rows x 2
    const int e = t >> 1;  // 0 .. 95
    *reinterpret_cast<uint4*>(dst + ((e >> 5) * 160 + ((e >> 1) & 15) * 10 + (e & 1) * 9) * 16) = make_uint4(0, 0, 0, 0);
  }
}

template <bool XBF, bool BN, bool ANY>
__device__ __forceinline__ void transform_kind(const uint8_t* raw, uint8_t* op, int t, const uint64_t (&sc)[4],
                                               const uint64_t (&sf)[4], int relu, const Geo& g, const Patch& pt) {
  if (!ANY) transform_px<XBF, BN, 0>(raw, op, t, sc, sf, relu, g, pt);
  else if (g.kind == C3_PATCH) transform_px<XBF, BN, C3_PATCH>(raw, op, t, sc, sf, relu, g, pt);
  else if (g.kind == C3_WHOLE) transform_px<XBF, BN, C3_WHOLE>(raw, op, t, sc, sf, relu, g, pt);
  else transform_px<XBF, BN, C3_SMALL>(raw, op, t, sc, sf, relu, g, pt);
}

template <int MODE, bool ANY>
__device__ __forceinline__ void c3_body(const ConvDesc* __restrict__ tab, const int* __restrict__ ts, int total,
                                        const Rings& rg, int32_t* status) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw0 = smem_u32(smem_raw);
  const uint32_t base = (raw0 + 1023u) & ~1023u;
  uint8_t* const gbase = smem_raw + (base - raw0);
  // [X ring | weight ring | output staging | reduction | operand ring | raw ring | Shared]
  // (the swizzled tiles first: every size before them is a multiple of 1024)
  const int off_w = rg.nx * rg.xb;
  uint8_t* const stage0 = gbase + off_w + rg.nu * rg.wb;
  uint8_t* const red0 = stage0 + kE * stage_bytes(MODE);
  const int off_op = off_w + rg.nu * rg.wb + kE * stage_bytes(MODE) + kGroups * kRedBytes;
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
      mbar_init(smem_u32(&sh.u_empty[s]), 1);
    }
    for (int s = 0; s < kMaxX; ++s) {
      mbar_init(smem_u32(&sh.x_full[s]), 1);
      mbar_init(smem_u32(&sh.x_empty[s]), 4);  // the tile's four epilogue warps
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
      Cursor cr(rg.nr), cu(rg.nu), cx(rg.nx);
      uint32_t ka = 0, u = 0, nx = 0;  // raw, weight and X slots issued
      bool ok = true;
      Geo g{};
      const void *ma = nullptr, *mx = nullptr;
      const uint8_t* wt = nullptr;
      uint32_t abytes = 0;
      int off = 0;
      for (Walk w(tab, ts, total); w.more() && ok; w.next(tab, ts)) {
        if (w.fresh) {
          const ConvDesc* d = w.d;
          g = geo<MODE, ANY>(d);
          ma = d->tma_a;
          mx = has_x<MODE>(d) ? d->tma_x : nullptr;
          wt = static_cast<const uint8_t*>(d->w);
          abytes = (uint32_t)(c3_raw_px(g.kind) * 16 * (MODE == FWD && d->x.dt == DT_BF16 ? 2 : 4));
          off = g.kind == C3_PATCH ? 1 : 0;
          tma_prefetch_map(ma);
          if (mx) tma_prefetch_map(mx);
        }
        const Patch p = patch(g, w.tm);
        const uint32_t wbytes = (uint32_t)c3_wt_bytes(g.n);
        const uint8_t* const wb = ANY ? wt + (size_t)w.tn * g.nk * wbytes : wt;  // the column block's weights
        for (int kt = 0; kt < g.nk; ++kt) {
          if (!mbar_wait(smem_u32(&sh.raw_empty[cr.s]), cr.ph ^ 1, abort_flag)) { ok = false; break; }
          const uint32_t full = smem_u32(&sh.raw_full[cr.s]);
          mbar_expect_tx(full, abytes);
          tma_load_4d(base + off_raw + cr.s * rg.rawb, ma, kt * 16, p.x0 - off, p.y0 - off, p.img, full);
          cr.next();
          ++ka;
          if (!mbar_wait(smem_u32(&sh.u_empty[cu.s]), cu.ph ^ 1, abort_flag)) { ok = false; break; }
          const uint32_t uf = smem_u32(&sh.u_full[cu.s]);
          mbar_expect_tx(uf, wbytes);
          bulk_load(base + off_w + cu.s * rg.wb, wb + (size_t)kt * wbytes, wbytes, uf);
          cu.next();
          ++u;
        }
        if (ok && mx != nullptr) {
          // (after the tile's k-steps: they must not wait for an earlier tile's epilogue)
          if (!mbar_wait(smem_u32(&sh.x_empty[cx.s]), cx.ph ^ 1, abort_flag)) { ok = false; break; }
          const uint32_t xf = smem_u32(&sh.x_full[cx.s]);
          mbar_expect_tx(xf, (uint32_t)(kTcBM * g.n * 2));
          tma_load_4d(base + cx.s * rg.xb, mx, ANY ? w.tn * g.n : 0, p.x0, p.y0, p.img, xf);
          cx.next();
          ++nx;
        }
      }
      if (!ok) { sh.abort_flag = 1; atomicExch(status, 3); }
      // the copies of the last slots issued must land before the CTA exits
      for (uint32_t i = ka > (uint32_t)rg.nr ? ka - rg.nr : 0; i < ka; ++i)
        mbar_wait_drain(smem_u32(&sh.raw_full[i % rg.nr]), (i / rg.nr) & 1);
      for (uint32_t i = u > (uint32_t)rg.nu ? u - rg.nu : 0; i < u; ++i)
        mbar_wait_drain(smem_u32(&sh.u_full[i % rg.nu]), (i / rg.nu) & 1);
      for (uint32_t i = nx > (uint32_t)rg.nx ? nx - rg.nx : 0; i < nx; ++i)
        mbar_wait_drain(smem_u32(&sh.x_full[i % rg.nx]), (i / rg.nx) & 1);
    }
    __syncwarp();
  } else if (warp == kMma) {
    // ================================================= MMA issuer
    if (elect_one()) {
      Cursor co(rg.no), cu(rg.nu), cx(rg.nx), cb(kAcc);
      bool ok = true, issued = false;
      Geo g{};
      bool hx = false;
      uint32_t idesc = 0;
      int rs = 0, ss = 1;  // pixels between the starts of tap rows and of taps
      for (Walk w(tab, ts, total); w.more() && ok; w.next(tab, ts), cb.next()) {
        if (w.fresh) {
          g = geo<MODE, ANY>(w.d);
          hx = has_x<MODE>(w.d);
          idesc = idesc_bf16(kTcBM, g.n);
          rs = g.kind == C3_PATCH ? 10 : !ANY || g.kind == C3_WHOLE ? 160 : 384;
          ss = ANY && g.kind == C3_SMALL ? 128 : 1;
        }
        const uint32_t tacc = tmem + cb.s * kAccCols;
        if (!mbar_wait(smem_u32(&sh.tempty[cb.s]), cb.ph ^ 1, abort_flag)) { ok = false; break; }
        for (int kt = 0; kt < g.nk; ++kt) {
          if (!mbar_wait(smem_u32(&sh.u_full[cu.s]), cu.ph, abort_flag)) { ok = false; break; }
          if (!mbar_wait(smem_u32(&sh.op_full[co.s]), co.ph, abort_flag)) { ok = false; break; }
          fence_after();
          // (descriptor starts count 16-byte units: one pixel, one weight row)
          const uint64_t ad = nosw_desc(base + off_op + co.s * rg.opb, c3_plane(g.kind), ANY && g.kind == C3_SMALL ? 128 : 160);
          const uint64_t bd = nosw_desc(base + off_w + cu.s * rg.wb, 9 * g.n * 16, 128);
#pragma unroll
          for (int tap = 0; tap < 9; ++tap) {
            const int r = MODE == FWD ? tap / 3 : 2 - tap / 3, s = MODE == FWD ? tap % 3 : 2 - tap % 3;
            mma_bf16(tacc, ad + r * rs + s * ss, bd + tap * g.n, idesc, (kt | tap) ? 1u : 0u);
          }
          issued = true;
          mma_commit(smem_u32(&sh.u_empty[cu.s]));
          mma_commit(smem_u32(&sh.op_empty[co.s]));
          co.next();
          cu.next();
        }
        // The tile's X, before its accumulator is announced: an epilogue group that has seen tfull finds
        // x_full of this tile complete, and the next phase of the slot needs the group's own arrivals -- a
        // parity wait of its own, two laps off, could not be mistaken for this one.
        if (ok && hx) {
          if (!mbar_wait(smem_u32(&sh.x_full[cx.s]), cx.ph, abort_flag)) { ok = false; break; }
          cx.next();
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
    for (Walk w(tab, ts, total); w.more(); w.next(tab, ts)) {
      const ConvDesc* d = w.d;
      if (w.fresh) {
        g = geo<MODE, ANY>(d);
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
          transform_kind<false, false, ANY>(raw, op, t, sc, sf, 0, g, p);
        } else if (xbf) {
          if (bn) transform_kind<true, true, ANY>(raw, op, t, sc, sf, relu, g, p);
          else transform_kind<true, false, ANY>(raw, op, t, sc, sf, 0, g, p);
        } else {
          if (bn) transform_kind<false, true, ANY>(raw, op, t, sc, sf, relu, g, p);
          else transform_kind<false, false, ANY>(raw, op, t, sc, sf, 0, g, p);
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
    Cursor cx(rg.nx), cb(kAcc);
    int turn = 0, sbuf = 0;
    const bool leader = elect_one();  // issues and waits for this warp's stores
    bool ok = true;
    Geo g{};
    EpiArgs ea{};
    for (Walk w(tab, ts, total); w.more(); w.next(tab, ts)) {
      if (w.fresh) {
        g = geo<MODE, ANY>(w.d);
        ea.load<MODE>(w.d);
      }
      const int xs = cx.s, b = cb.s;
      const uint32_t xph = cx.ph, bph = cb.ph;
      if (ea.hx) cx.next();
      cb.next();
      const bool mine = turn == eg;
      if (++turn == kGroups) turn = 0;
      if (!mine) continue;
      const int m0 = w.tm * kTcBM;
      if (ok) ok = mbar_wait(smem_u32(&sh.tfull[b]), bph, abort_flag);
      if (ok && ea.hx) ok = mbar_wait(smem_u32(&sh.x_full[xs]), xph, abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      float2* redw = es.red + es.rbuf * 256 + q * 64;
      if (ok) {
        fence_after();
        const uint32_t tacc = tmem + b * kAccCols + ((uint32_t)(q * 32) << 16);
        const uint8_t* x = gbase + xs * rg.xb;
        const uint32_t te = smem_u32(&sh.tempty[b]), ue = smem_u32(&sh.x_empty[xs]);
        const PatchDst<ANY> dst{patch(g, w.tm), g.kind, g.li};
        const int n0 = ANY ? w.tn * g.n : 0;
        if (MODE == FWD) {
          if (g.n == 64) unit_fwd<64>(ea, dst, tacc, q, lane, g.rows, m0, n0, x, st, redw, te, ue, leader);
          else if (g.n == 32) unit_fwd<32>(ea, dst, tacc, q, lane, g.rows, m0, n0, x, st, redw, te, ue, leader);
          else unit_fwd<16>(ea, dst, tacc, q, lane, g.rows, m0, n0, x, st, redw, te, ue, leader);
        } else {
          if (g.n == 64) unit_dgrad<64>(ea, dst, tacc, q, lane, g.rows, m0, n0, x, st, sbuf, redw, te, ue, leader);
          else if (g.n == 32) unit_dgrad<32>(ea, dst, tacc, q, lane, g.rows, m0, n0, x, st, sbuf, redw, te, ue, leader);
          else unit_dgrad<16>(ea, dst, tacc, q, lane, g.rows, m0, n0, x, st, sbuf, redw, te, ue, leader);
        }
      } else {
        sh.abort_flag = 1;
      }
      if (ea.stats) {
        float* p = ea.part + ((int64_t)w.tm * g.nt + (ANY ? w.tn * g.n : 0)) * 2;
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

template <bool ANY>
__global__ void __launch_bounds__(kThreads, 1) k_c3_fwd(const ConvDesc* __restrict__ tab, const int* __restrict__ ts,
                                                        int total, const Rings rg, int32_t* status) {
  c3_body<FWD, ANY>(tab, ts, total, rg, status);
}
template <bool ANY>
__global__ void __launch_bounds__(kThreads, 1) k_c3_dgrad(const ConvDesc* __restrict__ tab, const int* __restrict__ ts,
                                                          int total, const Rings rg, int32_t* status) {
  c3_body<DGRAD, ANY>(tab, ts, total, rg, status);
}

}  // namespace

cudaError_t launch_conv_c3(int mode, const ConvDesc* tab, const int* ts, int total, const C3Slots& s,
                           int32_t* status, cudaStream_t st, int max_ctas) {
  if (total <= 0) return cudaSuccess;
  if ((s.raw & 127) || (s.op & 127) || (s.wt & 1023) || (s.x & 1023) || s.raw <= 0 || s.op <= 0 || s.wt <= 0)
    return cudaErrorInvalidValue;
  Rings r;
  if (!(mode == FWD ? plan_rings<FWD>(s, r) : plan_rings<DGRAD>(s, r))) return cudaErrorInvalidValue;
  auto kern = mode == FWD ? (s.any ? k_c3_fwd<true> : k_c3_fwd<false>) : (s.any ? k_c3_dgrad<true> : k_c3_dgrad<false>);
  cudaError_t e = set_smem_attr_once((mode == FWD ? 17 : 18) + (s.any ? 2 : 0), reinterpret_cast<const void*>(kern), kSmemBudget);
  if (e != cudaSuccess) return e;
  const int sms = device_sm_count();
  int grid = total < sms ? total : sms;
  if (max_ctas > 0 && grid > max_ctas) grid = max_ctas;
  const int smem = (mode == FWD ? fixed_bytes<FWD>() : fixed_bytes<DGRAD>()) + rings_bytes(r);
  kern<<<grid, kThreads, smem, st>>>(tab, ts, total, r, status);
  return cudaGetLastError();
}

}  // namespace pnn
