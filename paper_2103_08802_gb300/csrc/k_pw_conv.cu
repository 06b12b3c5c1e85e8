// Grouped 1x1 stride-1 convolutions of the bottleneck stacks, forward and data
// gradient, on the 5th-generation tensor cores: the layers whose channel
// counts are so small (16 .. 256) that what the epilogue and the operand
// transform execute per element decides the time, not the MMA.
//
//   forward  y[m][n]  = res[m][n] + sum_k act(x)[m][k] * W[n][k],  bf16, and the BN statistics of y
//   dgrad    dx[m][n] (+)= sum_k dy[m][k] * Wt[n][k],  fp32, and the BN-backward sums of the BN in front
//
// One persistent CTA per SM walks the launch's items (an m-tile of 128 rows
// times a run of N units of BN = 64, 32 or 16 columns).  Roles:
//   producer    one thread: TMA boxes of raw A rows (a k-step: <= 64 channels)
//               into the raw ring, and per (k-step, unit) the weight box and
//               the unit's second operand X -- the residual (forward) or the
//               BN input h (data gradient) -- into the unit ring;
//   transform   T warps: raw rows -> BN scale/shift + ReLU (forward) -> bf16
//               operand, 128-byte-swizzled K-major.  A thread keeps one
//               8-channel chunk, so its scale and shift stay in registers;
//               packed fp32 pairs;
//   MMA         one thread, four accumulators of BN columns;
//   epilogue    groups of four warps (one per TMEM lane quarter), unit by unit:
//               the accumulator in one or two wide TMEM loads, X from shared
//               memory, the output staged in one swizzled tile per warp and
//               stored by TMA, the column sums from the staged tile with two
//               columns a lane.
// Against the per-16-column epilogue with residual rows gathered from global
// memory and scalar column sums (k_tc_conv.cu), an output element costs about
// a sixth of the instructions.  Bound by HBM latency and bandwidth, about half
// of the copy rate: grouped launches of the 8-subnetwork ResNet-1001 (batch
// 256, 64 px), before -> now: expand forward (16 -> 64 channels + residual +
// statistics) 218 -> 107 us, reduce forward 117 -> 73, reduce data gradient
// (+ BN-backward sums) 165 -> 128, expand data gradient 109 -> 88.
// Every wait is bounded (2 s); on expiry the CTA records status 3, stops,
// drains its copies and MMAs (bounded) and frees its TMEM.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "narrow_epilogue.cuh"
#include "pnn.h"
#include "pnn_internal.h"
#include "tc_pair.cuh"
#include "tc_ptx.cuh"

namespace pnn {
namespace {

using namespace tc;

constexpr int kRows = 128;
constexpr int kOpBytes = kRows * 128;      // one k-step's A operand (64 bf16 a row)
constexpr int kUnitB = 64 * 128;           // a unit's weight box: up to 64 rows x 64 bf16
constexpr int kMaxRing = 4;
constexpr int kAcc = 4;                    // TMEM accumulators of 64 columns
constexpr int kAccCols = 64;
constexpr int kSmemBudget = 227 * 1024;

// W = 1 (forward, every instance one k-step and N >= 64): the epilogue does
// most of the work, 2 transform + 12 epilogue warps; else 6 + 8.
template <int MODE, int W>
struct Roles {
  static constexpr int kT = W ? 2 : 6;
  static constexpr int kE = W ? 12 : 8;
  static constexpr int kProducer = 0, kMma = 1, kT0 = 2, kE0 = 2 + kT;
  static constexpr int kThreads = 32 * (2 + kT + kE);
  static constexpr int kGroups = kE / 4;
  static constexpr int kStage = stage_bytes(MODE);
};
static_assert(Roles<FWD, 0>::kE0 % 4 == 0 && Roles<FWD, 1>::kE0 % 4 == 0, "epilogue groups start at a TMEM lane quarter");

struct Shared {
  uint64_t raw_full[kMaxRing], raw_empty[kMaxRing];
  uint64_t op_full[kMaxRing], op_empty[kMaxRing];
  uint64_t u_full[kMaxRing], u_empty[kMaxRing];
  uint64_t tfull[kAcc], tempty[kAcc];
  uint64_t drain;
  uint32_t tmem;
  int abort_flag;
  float scale[kPwMaxC], shift[kPwMaxC];
};

// ring depths for a launch: raw and unit slot bytes follow from its instances
struct Rings {
  int nr, no, nu, rawb, ub;
};
__host__ __device__ inline int rings_bytes(const Rings& r) { return r.nr * r.rawb + r.no * kOpBytes + r.nu * r.ub; }

template <int MODE, int W>
constexpr int fixed_bytes() {
  return 1024 + (int)sizeof(Shared) + Roles<MODE, W>::kE * Roles<MODE, W>::kStage + Roles<MODE, W>::kGroups * kRedBytes;
}
template <int MODE, int W>
bool plan_rings(int rawb, int xb, Rings& r) {
  r = Rings{2, 2, 2, rawb, kUnitB + xb};
  const int avail = kSmemBudget - fixed_bytes<MODE, W>();
  if (rings_bytes(r) > avail) return false;
  // deepen the unit ring, then the raw ring, while they fit
  for (int* n : {&r.nu, &r.nr, &r.nu, &r.nr}) {
    if (*n >= kMaxRing) continue;
    ++*n;
    if (rings_bytes(r) > avail) --*n;
  }
  return true;
}

// two slots of each ring fit for the largest instance of pw_ok (64 fp32 channels a
// k-step, a second operand), so the launch of a planned group cannot fail
template <int MODE, int W>
constexpr bool fits() {
  return fixed_bytes<MODE, W>() + 2 * (pw_raw_bytes(kPwMaxC, 4) + kOpBytes + kUnitB + pw_x_bytes(64)) <= kSmemBudget;
}
static_assert(fits<FWD, 0>() && fits<FWD, 1>() && fits<DGRAD, 0>(), "two slots of each ring");

// what the roles need of an instance
struct Geo {
  int rows, ncols, kt, nkt, bn, spi, nsub;  // GEMM M, N, K; k-steps; unit columns; units an item, in all
};
template <int MODE>
__device__ __forceinline__ Geo geo(const ConvDesc* d) {
  Geo g;
  g.rows = d->B * d->H * d->W;
  g.ncols = MODE == FWD ? d->K : d->C;
  g.kt = MODE == FWD ? d->C : d->K;
  g.nkt = (g.kt + 63) >> 6;
  g.bn = pw_unit_cols(g.ncols);
  g.nsub = g.ncols / g.bn;
  g.spi = d->ntile_w / g.bn;
  return g;
}

// ------------------------------------------------------------ transform
// Rows of one k-step: raw [128][cw] (bf16 or fp32, dense) -> bf16 operand.
// Thread t of NT takes chunk t % nch (8 channels) of rows t / nch, + NT / nch ...
template <bool XBF, bool BN, int NT>
__device__ __forceinline__ void transform_rows(const uint8_t* __restrict__ raw, uint8_t* __restrict__ op, int lgn, int t,
                                               const float* __restrict__ scs, const float* __restrict__ sfs, int relu) {
  const int nch = 1 << lgn, cc = t & (nch - 1);
  const int rpitch = nch * (XBF ? 16 : 32);
  uint64_t sc[4], sf[4];
  if (BN) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 a = *reinterpret_cast<const float2*>(scs + cc * 8 + 2 * i);
      const float2 b = *reinterpret_cast<const float2*>(sfs + cc * 8 + 2 * i);
      sc[i] = pk2(a.x, a.y);
      sf[i] = pk2(b.x, b.y);
    }
  }
  const int step = NT >> lgn;
  const uint8_t* src = raw + cc * (XBF ? 16 : 32);
  // two rows a turn: both rows' loads first
  for (int r = t >> lgn; r < kRows; r += 2 * step) {
    const bool two = r + step < kRows;
    uint4 q[2][XBF ? 1 : 2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      if (e && !two) continue;
#pragma unroll
      for (int w = 0; w < (XBF ? 1 : 2); ++w)
        q[e][w] = *reinterpret_cast<const uint4*>(src + (r + e * step) * rpitch + 16 * w);
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      if (e && !two) continue;
      uint32_t o[4];
      if (XBF) {
        const uint32_t w[4] = {q[e][0].x, q[e][0].y, q[e][0].z, q[e][0].w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          o[i] = BN ? pack2(fma2(sc[i], bf2(w[i]), sf[i])) : w[i];
          if (BN && relu) o[i] = relu2(o[i]);
        }
      } else {
        const uint32_t* w = reinterpret_cast<const uint32_t*>(&q[e][0]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint64_t v = pk2(__uint_as_float(w[2 * i]), __uint_as_float(w[2 * i + 1]));
          o[i] = BN ? pack2(fma2(sc[i], v, sf[i])) : pack2(v);
          if (BN && relu) o[i] = relu2(o[i]);
        }
      }
      *reinterpret_cast<uint4*>(op + swz(r + e * step, cc)) = make_uint4(o[0], o[1], o[2], o[3]);
    }
  }
}

// where a warp's 32 rows of an output tile go
struct RowDst {
  int m0;
  __device__ __forceinline__ void put(const void* map, int n, int q, uint32_t src, bool add) const {
    if (add) tma_reduce_add_2d(map, n, m0 + q * 32, src);
    else tma_store_2d(map, n, m0 + q * 32, src);
  }
};

template <int MODE, int W>
__device__ __forceinline__ void pw_body(const ConvDesc* __restrict__ tab, const int* __restrict__ ts, int total,
                                        const Rings& rg, int32_t* status) {
  using R = Roles<MODE, W>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw0 = smem_u32(smem_raw);
  const uint32_t base = (raw0 + 1023u) & ~1023u;
  uint8_t* const gbase = smem_raw + (base - raw0);
  // [raw ring | operand ring | unit ring | output staging | reduction | Shared]
  const int off_op = rg.nr * rg.rawb;
  const int off_u = off_op + rg.no * kOpBytes;
  const int off_st = off_u + rg.nu * rg.ub;
  uint8_t* const stage0 = gbase + off_st;
  uint8_t* const red0 = stage0 + R::kE * R::kStage;
  Shared& sh = *reinterpret_cast<Shared*>(red0 + R::kGroups * kRedBytes);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kMaxRing; ++s) {
      mbar_init(smem_u32(&sh.raw_full[s]), 1);
      mbar_init(smem_u32(&sh.raw_empty[s]), R::kT);
      mbar_init(smem_u32(&sh.op_full[s]), R::kT);
      mbar_init(smem_u32(&sh.op_empty[s]), 1);
      mbar_init(smem_u32(&sh.u_full[s]), 1);
      // the MMA's commit and the readers of X: the unit's four epilogue warps, or (no X) the MMA thread for them
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
  if (warp == R::kMma) tmem_alloc(smem_u32(&sh.tmem), kAcc * kAccCols);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = sh.tmem;
  volatile int* abort_flag = &sh.abort_flag;

  if (warp == R::kProducer) {
    // ================================================= TMA producer
    if (elect_one()) {
      Cursor cr(rg.nr), cu(rg.nu);
      uint32_t ka = 0, u = 0;  // k-steps and units issued
      bool ok = true;
      Geo g{};
      const void *ma = nullptr, *mb = nullptr, *mx = nullptr;
      uint32_t abytes = 0;
      for (Walk w(tab, ts, total); w.more() && ok; w.next(tab, ts)) {
        if (w.fresh) {
          const ConvDesc* d = w.d;
          g = geo<MODE>(d);
          ma = d->tma_a;
          mb = d->tma_b;
          mx = has_x<MODE>(d) ? d->tma_x : nullptr;
          abytes = (uint32_t)(kRows * min(g.kt, 64) * (MODE == FWD && d->x.dt == DT_BF16 ? 2 : 4));
          tma_prefetch_map(ma);
          tma_prefetch_map(mb);
          if (mx) tma_prefetch_map(mx);
        }
        const int m0 = w.tm * kRows, sub0 = w.tn * g.spi, sub1 = min(g.nsub, sub0 + g.spi);
        for (int kt = 0; kt < g.nkt && ok; ++kt) {
          if (!mbar_wait(smem_u32(&sh.raw_empty[cr.s]), cr.ph ^ 1, abort_flag)) { ok = false; break; }
          const uint32_t full = smem_u32(&sh.raw_full[cr.s]);
          mbar_expect_tx(full, abytes);
          tma_load_2d(base + cr.s * rg.rawb, ma, kt * 64, m0, full);
          cr.next();
          ++ka;
          for (int sub = sub0; sub < sub1; ++sub) {
            if (!mbar_wait(smem_u32(&sh.u_empty[cu.s]), cu.ph ^ 1, abort_flag)) { ok = false; break; }
            const uint32_t uf = smem_u32(&sh.u_full[cu.s]);
            const uint32_t slot = base + off_u + cu.s * rg.ub;
            const bool x = mx != nullptr && kt == g.nkt - 1;
            mbar_expect_tx(uf, (uint32_t)(g.bn * 128 + (x ? kRows * g.bn * 2 : 0)));
            tma_load_2d(slot, mb, kt * 64, sub * g.bn, uf);
            if (x) tma_load_2d(slot + kUnitB, mx, sub * g.bn, m0, uf);
            cu.next();
            ++u;
          }
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
  } else if (warp == R::kMma) {
    // ================================================= MMA issuer
    if (elect_one()) {
      Cursor co(rg.no), cu(rg.nu), cb(kAcc);
      bool ok = true, issued = false;
      Geo g{};
      bool hx = false;
      uint32_t idesc = 0;
      for (Walk w(tab, ts, total); w.more() && ok; w.next(tab, ts)) {
        if (w.fresh) {
          g = geo<MODE>(w.d);
          hx = has_x<MODE>(w.d);
          idesc = idesc_bf16(kRows, g.bn);
        }
        const int sub0 = w.tn * g.spi, sub1 = min(g.nsub, sub0 + g.spi);
        for (int kt = 0; kt < g.nkt && ok; ++kt) {
          if (!mbar_wait(smem_u32(&sh.op_full[co.s]), co.ph, abort_flag)) { ok = false; break; }
          const uint32_t a_addr = base + off_op + co.s * kOpBytes;
          const int ksub = min(4, (g.kt - kt * 64) >> 4);
          for (int sub = sub0; sub < sub1; ++sub) {
            // (several k-steps go with a single unit an item: cb stays on its accumulator until the last)
            if (kt == 0 && !mbar_wait(smem_u32(&sh.tempty[cb.s]), cb.ph ^ 1, abort_flag)) { ok = false; break; }
            if (!mbar_wait(smem_u32(&sh.u_full[cu.s]), cu.ph, abort_flag)) { ok = false; break; }
            fence_after();
            const uint32_t b_addr = base + off_u + cu.s * rg.ub;
            const uint32_t tacc = tmem + cb.s * kAccCols;
            for (int kk = 0; kk < ksub; ++kk)
              mma_bf16(tacc, sw128_desc(a_addr + kk * 32), sw128_desc(b_addr + kk * 32), idesc, (kt | kk) ? 1u : 0u);
            issued = true;
            if (!(hx && kt == g.nkt - 1)) mbar_arrive_n(smem_u32(&sh.u_empty[cu.s]), 4);
            mma_commit(smem_u32(&sh.u_empty[cu.s]));
            cu.next();
            if (kt == g.nkt - 1) {
              mma_commit(smem_u32(&sh.tfull[cb.s]));
              cb.next();
            }
          }
          if (ok) mma_commit(smem_u32(&sh.op_empty[co.s]));
          co.next();
        }
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
  } else if (warp < R::kE0) {
    // ================================================= transform
    // Every transform thread walks every k-step (they meet at named barrier 1
    // when the instance changes): a thread whose wait fails stops working but
    // keeps walking.
    constexpr int NT = 32 * R::kT;
    const int t = threadIdx.x - 32 * R::kT0;
    Cursor cr(rg.nr), co(rg.no);
    bool ok = true;
    Geo g{};
    bool bn = false, xbf = false;
    int relu = 0, lgn = 0;
    for (Walk w(tab, ts, total); w.more(); w.next(tab, ts)) {
      const ConvDesc* d = w.d;
      if (w.fresh) {
        g = geo<MODE>(d);
        bn = MODE == FWD && d->x.scale != nullptr;
        xbf = MODE == FWD && d->x.dt == DT_BF16;
        relu = bn ? d->x.relu : 0;
        lgn = 28 - __clz(min(g.kt, 64));  // log2 of the 8-channel chunks a row
      }
      if (bn && w.fresh) {
        asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");  // all are past the previous instance
        for (int c = t; c < g.kt; c += NT) {
          sh.scale[c] = __ldg(d->x.scale + c);
          sh.shift[c] = __ldg(d->x.shift + c);
        }
        asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");
      }
      for (int kt = 0; kt < g.nkt; ++kt, cr.next(), co.next()) {
        const int sr = cr.s, so = co.s;
        if (ok) ok = mbar_wait(smem_u32(&sh.raw_full[sr]), cr.ph, abort_flag);
        if (ok) ok = mbar_wait(smem_u32(&sh.op_empty[so]), co.ph ^ 1, abort_flag);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) { sh.abort_flag = 1; continue; }
        const uint8_t* raw = gbase + sr * rg.rawb;
        uint8_t* op = gbase + off_op + so * kOpBytes;
        if (MODE == DGRAD) {
          transform_rows<false, false, NT>(raw, op, lgn, t, nullptr, nullptr, 0);
        } else if (xbf) {
          if (bn) transform_rows<true, true, NT>(raw, op, lgn, t, sh.scale + kt * 64, sh.shift + kt * 64, relu);
          else transform_rows<true, false, NT>(raw, op, lgn, t, nullptr, nullptr, 0);
        } else {
          if (bn) transform_rows<false, true, NT>(raw, op, lgn, t, sh.scale + kt * 64, sh.shift + kt * 64, relu);
          else transform_rows<false, false, NT>(raw, op, lgn, t, nullptr, nullptr, 0);
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(smem_u32(&sh.raw_empty[sr]));
          mbar_arrive(smem_u32(&sh.op_full[so]));
        }
      }
    }
    if (!ok) { sh.abort_flag = 1; atomicExch(status, 3); }
  } else {
    // ================================================= epilogue
    const int ew = warp - R::kE0, q = warp & 3, eg = ew >> 2;
    uint8_t* const st = stage0 + ew * R::kStage;
    EpiState es{reinterpret_cast<float2*>(red0 + eg * kRedBytes), 0, 2 + eg};
    Cursor cu(rg.nu), cb(kAcc);
    int turn = 0, sbuf = 0;
    const bool leader = elect_one();  // issues and waits for this warp's stores
    bool ok = true;
    Geo g{};
    EpiArgs ea{};
    for (Walk w(tab, ts, total); w.more(); w.next(tab, ts)) {
      if (w.fresh) {
        g = geo<MODE>(w.d);
        ea.load<MODE>(w.d);
      }
      const int m0 = w.tm * kRows, sub0 = w.tn * g.spi, sub1 = min(g.nsub, sub0 + g.spi);
      for (int sub = sub0; sub < sub1; ++sub) {
        // the unit's last k-step holds X (one unit a k-step: sub1 - sub0 == 1 when nkt > 1)
        for (int i = 1; i < g.nkt; ++i) cu.next();
        const int us = cu.s, b = cb.s;
        const uint32_t uph = cu.ph, bph = cb.ph;
        cu.next();
        cb.next();
        const bool mine = turn == eg;
        if (++turn == R::kGroups) turn = 0;
        if (!mine) continue;
        if (ok) ok = mbar_wait(smem_u32(&sh.tfull[b]), bph, abort_flag);
        if (ok && ea.hx) ok = mbar_wait(smem_u32(&sh.u_full[us]), uph, abort_flag);
        ok = __all_sync(0xffffffffu, ok);
        const int n0 = sub * g.bn;
        float2* redw = es.red + es.rbuf * 256 + q * 64;
        if (ok) {
          fence_after();
          const uint32_t tacc = tmem + b * kAccCols + ((uint32_t)(q * 32) << 16);
          const uint8_t* x = gbase + off_u + us * rg.ub + kUnitB;
          const uint32_t te = smem_u32(&sh.tempty[b]), ue = smem_u32(&sh.u_empty[us]);
          const RowDst dst{m0};
          if (MODE == FWD) {
            if (g.bn == 64) unit_fwd<64>(ea, dst, tacc, q, lane, g.rows, m0, n0, x, st, redw, te, ue, leader);
            else if (g.bn == 32) unit_fwd<32>(ea, dst, tacc, q, lane, g.rows, m0, n0, x, st, redw, te, ue, leader);
            else unit_fwd<16>(ea, dst, tacc, q, lane, g.rows, m0, n0, x, st, redw, te, ue, leader);
          } else {
            if (g.bn == 64) unit_dgrad<64>(ea, dst, tacc, q, lane, g.rows, m0, n0, x, st, sbuf, redw, te, ue, leader);
            else if (g.bn == 32) unit_dgrad<32>(ea, dst, tacc, q, lane, g.rows, m0, n0, x, st, sbuf, redw, te, ue, leader);
            else unit_dgrad<16>(ea, dst, tacc, q, lane, g.rows, m0, n0, x, st, sbuf, redw, te, ue, leader);
          }
        } else {
          sh.abort_flag = 1;
        }
        if (ea.stats) {
          float* p = ea.part + ((int64_t)w.tm * g.ncols + n0) * 2;
          if (g.bn == 64) merge_partials<MODE, 64>(es, ok, q, lane, g.rows, m0, p);
          else if (g.bn == 32) merge_partials<MODE, 32>(es, ok, q, lane, g.rows, m0, p);
          else merge_partials<MODE, 16>(es, ok, q, lane, g.rows, m0, p);
        }
      }
    }
    // the output stores must complete before the CTA exits
    if (leader) bulk_wait_all();
    __syncwarp();
    if (!ok) { sh.abort_flag = 1; atomicExch(status, 3); }
  }
  fence_before();
  __syncthreads();
  if (warp == R::kMma) {
    fence_after();
    tmem_dealloc(tmem, kAcc * kAccCols);
  }
}

#define PNN_PW_KERNEL(NAME, MODE, W)                                                                                \
  __global__ void __launch_bounds__(Roles<MODE, W>::kThreads, 1)                                                    \
      NAME(const ConvDesc* __restrict__ tab, const int* __restrict__ ts, int total, const Rings rg,                 \
           int32_t* status) {                                                                                       \
    pw_body<MODE, W>(tab, ts, total, rg, status);                                                                   \
  }
PNN_PW_KERNEL(k_pw_fwd, FWD, 0)
PNN_PW_KERNEL(k_pw_fwd_w, FWD, 1)
PNN_PW_KERNEL(k_pw_dgrad, DGRAD, 0)

template <int MODE, int W>
cudaError_t launch(void (*kern)(const ConvDesc*, const int*, int, const Rings, int32_t*), int slot,
                   const ConvDesc* tab, const int* ts, int total, int raw_bytes, int x_bytes,
                   int32_t* status, cudaStream_t st, int max_ctas) {
  Rings r;
  if (!plan_rings<MODE, W>(raw_bytes, x_bytes, r)) return cudaErrorInvalidValue;
  cudaError_t e = set_smem_attr_once(slot, reinterpret_cast<const void*>(kern), kSmemBudget);
  if (e != cudaSuccess) return e;
  const int sms = device_sm_count();
  int grid = total < sms ? total : sms;
  if (max_ctas > 0 && grid > max_ctas) grid = max_ctas;
  const int smem = fixed_bytes<MODE, W>() + rings_bytes(r);
  kern<<<grid, Roles<MODE, W>::kThreads, smem, st>>>(tab, ts, total, r, status);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_conv_pw(int mode, int wide, const ConvDesc* tab, const int* ts, int total, int raw_bytes,
                           int x_bytes, int32_t* status, cudaStream_t st, int max_ctas) {
  if (total <= 0) return cudaSuccess;
  if (raw_bytes <= 0 || (raw_bytes & 1023) || x_bytes < 0 || (x_bytes & 1023)) return cudaErrorInvalidValue;
  if (mode == DGRAD)
    return launch<DGRAD, 0>(k_pw_dgrad, 14, tab, ts, total, raw_bytes, x_bytes, status, st, max_ctas);
  return wide ? launch<FWD, 1>(k_pw_fwd_w, 13, tab, ts, total, raw_bytes, x_bytes, status, st, max_ctas)
              : launch<FWD, 0>(k_pw_fwd, 12, tab, ts, total, raw_bytes, x_bytes, status, st, max_ctas);
}

}  // namespace pnn
