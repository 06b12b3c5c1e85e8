// CUDA-core kernels of the parareal training step: implicit-GEMM convolution
// (forward, data gradient, weight gradient) used in fp32 check mode, and every
// non-convolution op of the step (BN statistics and backward, elementwise
// correction/residual ops, pooling, head, loss, SGD) used in both precisions.
//
// Every kernel is "grouped": one launch covers a list of independent problem
// instances (typically the same layer position of all N fine subnetworks,
// Algorithm 1's parallel loop), each CTA finds its instance from a tile prefix.
// All reductions run in a fixed order so that results are bit-reproducible.
//
// Fixed order: an fp32 network (check mode) further keeps the order of its sums
// from version to version, whatever the tiles and splits of the kernels are.
// The last bit of a BN statistic decides whether a pre-activation next to zero
// passes the ReLU, and one that flips moves the gradients by 1e-5 to 1e-3, far
// above the 1e-7 of a rounding.  The order: conv and FC outputs one fused
// multiply-add after another; BN partials over 256, 128 or 64 rows (layers of at
// most 16, at most 32, more channels) in 16 row groups, or of an elementwise sum
// over 64 rows in 256 / C; their combination as in tile_moments_fixed; weight
// gradients over the pixels of a split, BN-backward sums over the rows of tiles of
// bnb_fixed_rows, average pool and bias gradients over pixels and images.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <mutex>

#include "pnn_internal.h"
#include "tc_pair.cuh"

namespace pnn {

// ---------------------------------------------------------------- helpers
__device__ __forceinline__ float ldv(const void* p, int dt, int64_t i) {
  return dt == DT_F32 ? __ldg(reinterpret_cast<const float*>(p) + i)
                      : __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(p)[i]);
}
__device__ __forceinline__ float rnd(int dt, float v) {
  return dt == DT_BF16 ? __bfloat162float(__float2bfloat16_rn(v)) : v;
}
__device__ __forceinline__ void stv(void* p, int dt, int64_t i, float v) {
  if (dt == DT_F32) reinterpret_cast<float*>(p)[i] = v;
  else reinterpret_cast<__nv_bfloat16*>(p)[i] = __float2bfloat16_rn(v);
}
__device__ __forceinline__ float ld_src(const Src& s, int64_t i, int c) {
  float v = ldv(s.ptr, s.dt, i);
  if (s.scale) {
    v = fmaf(__ldg(s.scale + c), v, __ldg(s.shift + c));
    if (s.relu) v = fmaxf(v, 0.f);
  }
  return v;
}
// index of the instance that owns CTA b: the largest i with tstart[i] <= b
// (every thread of the block calls it with the same b: up to 32 instances
// the warp reads the starts at once and counts those <= b -- one dependent
// load instead of log2(n) -- else a binary search)
__device__ __forceinline__ int find_instance(const int* tstart, int n, int b) {
  if (n <= 32) {
    const int lane = threadIdx.x & 31;
    const bool le = lane < n && __ldg(tstart + lane) <= b;
    return __popc(__ballot_sync(0xffffffffu, le)) - 1;
  }
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (__ldg(tstart + mid) <= b) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// ---------------------------------------------------------------- conv fwd
// The CUDA-core convolutions (fp32 check mode, and channel counts the tensor
// cores do not take) run 16-wide steps over the contraction index with the
// next step's global loads in registers while the current one is multiplied
// from shared memory.  A thread loads one contraction index k for every 16th
// row, so (r, s, c) is stepped, not divided, and each row's coordinates come
// from a table formed once per CTA.  (With divisions per element and no loads
// in flight ahead, one fp32 3x3 layer of two subnetworks with 16 channels at
// batch 8 took 86 us forward, 105 us for its data and 81 us for its weight
// gradient; now 20, 18 and 26 us.)
struct TapStep {  // contraction index k = (r * S + s) * C + c
  int r, s, c;
  __device__ __forceinline__ TapStep(int k, int S, int C) {
    c = k % C;
    const int rs = k / C;
    s = rs % S;
    r = rs / S;
  }
  __device__ __forceinline__ void advance(int n, int S, int C) {
    c += n;
    while (c >= C) {
      c -= C;
      if (++s == S) { s = 0; ++r; }
    }
  }
};
constexpr int kRowOutside = -0x4000;  // a row coordinate no tap brings into an image

// BN partial (mean, M2) of a thread's rows m0 + 16 i < M, i < tm: two passes
template <typename Get>
__device__ __forceinline__ float2 row_moments(int tm, int m0, int M, Get v) {
  int cnt = 0;
  float s1 = 0.f, m2 = 0.f;
#pragma unroll
  for (int i = 0; i < tm; ++i)
    if (m0 + 16 * i < M) {
      s1 += v(i);
      ++cnt;
    }
  const float mean = cnt > 0 ? s1 / (float)cnt : 0.f;
#pragma unroll
  for (int i = 0; i < tm; ++i)
    if (m0 + 16 * i < M) m2 = fmaf(v(i) - mean, v(i) - mean, m2);
  return make_float2(mean, m2);
}
// the partial of the rows m0 .. m0 + 16 tm - 1 from its 16 row groups, in order
template <typename Get>
__device__ __forceinline__ void merge_row_groups(int tm, int m0, int M, Get red, float* out) {
  float n = 0.f, mean = 0.f, m2 = 0.f;
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    const int cr = min(tm, max(0, (M - m0 - r + 15) >> 4));  // rows m0 + r + 16 i < M, i < tm
    const float2 v = red(r);
    chan_merge(n, mean, m2, (float)cr, v.x, v.y);
  }
  out[0] = mean;
  out[1] = m2;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// *p of CTA `rank` of the cluster (p: this CTA's shared memory)
__device__ __forceinline__ float ld_cluster(const float* p, uint32_t rank) {
  uint32_t at;
  float x;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(x) : "r"(at));
  return x;
}

// Y[m][k] = sum_{r,s,c} act(X)[n, p*st+r-pad, q*st+s-pad, c] * W[k][r][s][c] (+ res[m][k])
// CL: CTAs of a cluster, whose rows form one partial of the BN statistics.  (With 256
// rows a CTA, as the fixed order wants them, a batch of 8 at 32 x 32 occupies 32 SMs.)
template <int BM, int BN, int CL>
__device__ __forceinline__ void conv_fwd_body(const ConvDesc* __restrict__ tab, const int* __restrict__ tstart, int n) {
  constexpr int BK = 16, TM = BM / 16, TN = BN / 16;
  __shared__ float As[2][BK][BM + 4];
  __shared__ float Bs[2][BK][BN + 4];
  __shared__ float red[16][BN][2];
  __shared__ float quad[CL == 1 ? 1 : BM][CL == 1 ? 1 : BN + 1];
  __shared__ int rowp[BM], rowh[BM], roww[BM];  // pixel index of tap (0, 0), its row and column
  const int inst = find_instance(tstart, n, blockIdx.x);
  const ConvDesc d = tab[inst];
  const int t = blockIdx.x - tstart[inst];
  const int tm = t % d.mtiles, tn = t / d.mtiles;
  const int M = d.B * d.P * d.Q, Kt = d.R * d.S * d.C;
  const int m0 = tm * BM, n0 = tn * BN;
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  for (int mm = tid; mm < BM; mm += 256) {
    const int m = m0 + mm, q = m % d.Q, tmp = m / d.Q, pp = tmp % d.P, nb = tmp / d.P;
    const int h = pp * d.stride - d.pad, w = q * d.stride - d.pad;
    rowh[mm] = m < M ? h : kRowOutside;
    roww[mm] = w;
    rowp[mm] = (nb * d.H + h) * d.W + w;
  }
  __syncthreads();
  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;

  const int kk = tx;  // this thread's index within a step
  TapStep ts(kk, d.S, d.C);
  float ra[TM], rb[TN];
  unsigned in = 0;
  float sc = 1.f, sf = 0.f;
  auto load = [&](int k0) {
    const int k = k0 + kk;
    in = 0;
    if (k < Kt) {
      if (d.x.scale) { sc = __ldg(d.x.scale + ts.c); sf = __ldg(d.x.shift + ts.c); }
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const int mm = ty + 16 * i;
        const int h = rowh[mm] + ts.r, w = roww[mm] + ts.s;
        ra[i] = 0.f;
        if (h >= 0 && h < d.H && w >= 0 && w < d.W) {
          in |= 1u << i;
          ra[i] = ldv(d.x.ptr, d.x.dt, (int64_t)(rowp[mm] + ts.r * d.W + ts.s) * d.C + ts.c);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int co = n0 + ty + 16 * j;
      rb[j] = k < Kt && co < d.K ? ldv(d.w, d.w_dt, (int64_t)co * Kt + k) : 0.f;
    }
    ts.advance(BK, d.S, d.C);
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      float v = 0.f;
      if ((in >> i) & 1) {
        v = ra[i];
        if (d.x.scale) {
          v = fmaf(sc, v, sf);
          if (d.x.relu) v = fmaxf(v, 0.f);
        }
      }
      As[buf][kk][ty + 16 * i] = d.op_bf16 ? rnd(DT_BF16, v) : v;
    }
#pragma unroll
    for (int j = 0; j < TN; ++j) Bs[buf][kk][ty + 16 * j] = rb[j];
  };
  load(0);
  store(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < Kt; k0 += BK) {
    const bool more = k0 + BK < Kt;
    if (more) load(k0 + BK);
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      float a[TM], b[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = As[buf][k][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < TN; ++j) b[j] = Bs[buf][k][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    if (more) store(buf ^ 1);
    __syncthreads();
    buf ^= 1;
  }
  // epilogue: residual, store, BN partials of the stored value
#pragma unroll
  for (int j = 0; j < TN; ++j) {
    const int co = n0 + tx + 16 * j;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int m = m0 + ty + 16 * i;
      if (m < M && co < d.K) {
        const int64_t o = (int64_t)m * d.K + co;
        float v = acc[i][j];
        if (d.res) v += ldv(d.res, d.res_dt, o);
        if (d.res2[0]) v = fmaf(d.res2_c[0], ldv(d.res2[0], d.res2_dt[0], o), v);
        if (d.res2[1]) v = fmaf(d.res2_c[1], ldv(d.res2[1], d.res2_dt[1], o), v);
        v = rnd(d.y_dt, v);
        stv(d.y, d.y_dt, o, v);
        acc[i][j] = v;
      }
    }
  }
  if (!d.stats) return;
  if (CL == 1) {
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const float2 v = row_moments(TM, m0 + ty, M, [&](int i) { return acc[i][j]; });
      red[ty][tx + 16 * j][0] = v.x;
      red[ty][tx + 16 * j][1] = v.y;
    }
    __syncthreads();
    for (int nn = tid; nn < BN; nn += 256)
      if (n0 + nn < d.K)
        merge_row_groups(TM, m0, M, [&](int r) { return make_float2(red[r][nn][0], red[r][nn][1]); },
                         d.stats + ((int64_t)tm * d.K + n0 + nn) * 2);
  } else {
    // the cluster's first CTA reads the others' rows
    static_assert(CL == 1 || BN == 16, "a column a thread");
#pragma unroll
    for (int i = 0; i < TM; ++i) quad[CL == 1 ? 0 : ty + 16 * i][CL == 1 ? 0 : tx] = acc[i][0];
    cluster_sync();
    if (tm % CL == 0) {
      float v[TM * CL];
#pragma unroll
      for (int i = 0; i < TM * CL; ++i)
        v[i] = i < TM ? acc[i % TM][0] : ld_cluster(&quad[CL == 1 ? 0 : ty + 16 * (i % TM)][CL == 1 ? 0 : tx], i / TM);
      const float2 s = row_moments(TM * CL, m0 + ty, M, [&](int i) { return v[i]; });
      red[ty][tx][0] = s.x;
      red[ty][tx][1] = s.y;
      __syncthreads();
      if (tid < BN && n0 + tid < d.K)
        merge_row_groups(TM * CL, m0, M, [&](int r) { return make_float2(red[r][tid][0], red[r][tid][1]); },
                         d.stats + ((int64_t)(tm / CL) * d.K + n0 + tid) * 2);
    }
    cluster_sync();  // a CTA's shared memory stays until it has been read
  }
}
template <int BM, int BN>
__global__ void __launch_bounds__(256) k_conv_fwd(const ConvDesc* __restrict__ tab,
                                                  const int* __restrict__ tstart, int n) {
  conv_fwd_body<BM, BN, 1>(tab, tstart, n);
}
__global__ void __cluster_dims__(kQuad, 1, 1) __launch_bounds__(256)
    k_conv_fwd_quad(const ConvDesc* __restrict__ tab, const int* __restrict__ tstart, int n) {
  conv_fwd_body<64, 16, kQuad>(tab, tstart, n);
}

// ---------------------------------------------------------------- conv dgrad
// dX[m=(n,h,w)][c] (+)= sum_{r,s,k} dY[n, (h+pad-r)/st, (w+pad-s)/st, k] * W[k][r][s][c]
// (terms whose division is inexact or out of range are zero)
template <int BM, int BN>
__global__ void __launch_bounds__(256) k_conv_dgrad(const ConvDesc* __restrict__ tab,
                                                    const int* __restrict__ tstart, int n) {
  constexpr int BK = 16, TM = BM / 16, TN = BN / 16;
  __shared__ float As[2][BK][BM + 4];
  __shared__ float Bs[2][BK][BN + 4];
  __shared__ int rown[BM], rowh[BM], roww[BM];  // image, row + pad, column + pad
  const int inst = find_instance(tstart, n, blockIdx.x);
  const ConvDesc d = tab[inst];
  const int t = blockIdx.x - tstart[inst];
  const int tm = t % d.mtiles, tn = t / d.mtiles;
  const int M = d.B * d.H * d.W, Kt = d.R * d.S * d.K;
  const int m0 = tm * BM, n0 = tn * BN;
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  for (int mm = tid; mm < BM; mm += 256) {
    const int m = m0 + mm, w = m % d.W, tmp = m / d.W, h = tmp % d.H;
    rown[mm] = tmp / d.H;
    rowh[mm] = m < M ? h + d.pad : kRowOutside;
    roww[mm] = w + d.pad;
  }
  __syncthreads();
  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;
  const int kk = tx;  // this thread's A index within a step
  const int sl = d.stride - 1;  // stride 1 or 2: log2, and the mask of an inexact division
  TapStep ts(kk, d.S, d.K), tb(ty, d.S, d.K);  // B is loaded with c across the lanes: its k is k0 + ty
  float ra[TM], rb[TN];
  auto load = [&](int k0) {
    const int k = k0 + kk;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int mm = ty + 16 * i;
      const int pn = rowh[mm] - ts.r, qn = roww[mm] - ts.s;
      const int p = pn >> sl, q = qn >> sl;
      ra[i] = 0.f;
      if (k < Kt && pn >= 0 && qn >= 0 && ((pn | qn) & sl) == 0 && p < d.P && q < d.Q)
        ra[i] = __ldg(d.dy + ((int64_t)(rown[mm] * d.P + p) * d.Q + q) * d.K + ts.c);
    }
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int c = n0 + tx + 16 * j;
      rb[j] = k0 + ty < Kt && c < d.C ? ldv(d.w, d.w_dt, ((int64_t)tb.c * d.R * d.S + tb.r * d.S + tb.s) * d.C + c) : 0.f;
    }
    ts.advance(BK, d.S, d.K);
    tb.advance(BK, d.S, d.K);
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int i = 0; i < TM; ++i) As[buf][kk][ty + 16 * i] = d.op_bf16 ? rnd(DT_BF16, ra[i]) : ra[i];
#pragma unroll
    for (int j = 0; j < TN; ++j) Bs[buf][ty][tx + 16 * j] = rb[j];
  };
  load(0);
  store(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < Kt; k0 += BK) {
    const bool more = k0 + BK < Kt;
    if (more) load(k0 + BK);
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      float a[TM], b[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = As[buf][k][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < TN; ++j) b[j] = Bs[buf][k][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    if (more) store(buf ^ 1);
    __syncthreads();
    buf ^= 1;
  }
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int m = m0 + ty + 16 * i;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int c = n0 + tx + 16 * j;
      if (m < M && c < d.C) {
        const int64_t o = (int64_t)m * d.C + c;
        d.dx[o] = d.accumulate ? d.dx[o] + acc[i][j] : acc[i][j];
      }
    }
  }
}

// ---------------------------------------------------------------- conv wgrad
// part[split][k][(r,s,c)] = sum_{m in split} dY[m][k] * act(X)[n, p*st+r-pad, q*st+s-pad, c]
// BM = 64 output channels a tile, or 16 for layers that have no more
template <int BM>
__global__ void __launch_bounds__(256) k_conv_wgrad(const ConvDesc* __restrict__ tab,
                                                    const int* __restrict__ tstart, int n) {
  constexpr int BN = kWgradBN, BK = kWgradBK, TM = BM / 16, TN = BN / 16;
  static_assert(BN == 64 && BK == 16, "a thread loads one (r, s, c) and every fourth pixel of a step");
  __shared__ float As[2][BK][BM + 4];
  __shared__ float Bs[2][BK][BN + 4];
  const int inst = find_instance(tstart, n, blockIdx.x);
  const ConvDesc d = tab[inst];
  int t = blockIdx.x - tstart[inst];
  const int tm = t % d.mtiles;
  t /= d.mtiles;
  const int tn = t % d.ntiles, split = t / d.ntiles;
  const int RSC = d.R * d.S * d.C, Mp = d.B * d.P * d.Q;
  const int m0 = tm * BM, n0 = tn * BN;
  const int p_begin = split * d.pix_per_split;
  const int p_end = min(Mp, p_begin + d.pix_per_split);
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;
  // B: column jn = tid % 64 (its tap and channel fixed), pixels tid / 64 + 4 i
  const int jn = tid % BN, pk = tid / BN;
  const bool jin = n0 + jn < RSC;
  const TapStep ts(jin ? n0 + jn : 0, d.S, d.C);
  float sc = 1.f, sf = 0.f;
  if (d.x.scale) { sc = __ldg(d.x.scale + ts.c); sf = __ldg(d.x.shift + ts.c); }
  // (image, row, column) of output pixel k0 + pk + 4 i, stepped
  int nb[4], ph[4], pw[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int pix = p_begin + pk + 4 * i;
    pw[i] = pix % d.Q;
    const int tmp = pix / d.Q;
    ph[i] = tmp % d.P;
    nb[i] = tmp / d.P;
  }
  constexpr int NA = BM * BK / 256;
  float ra[NA], rb[4];
  unsigned in = 0;
  auto load = [&](int k0) {
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      const int mm = (tid + 256 * i) % BM, pix = k0 + (tid + 256 * i) / BM;
      ra[i] = m0 + mm < d.K && pix < p_end ? __ldg(d.dy + (int64_t)pix * d.K + m0 + mm) : 0.f;
    }
    in = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int h = ph[i] * d.stride + ts.r - d.pad, w = pw[i] * d.stride + ts.s - d.pad;
      rb[i] = 0.f;
      if (jin && k0 + pk + 4 * i < p_end && h >= 0 && h < d.H && w >= 0 && w < d.W) {
        in |= 1u << i;
        rb[i] = ldv(d.x.ptr, d.x.dt, ((int64_t)(nb[i] * d.H + h) * d.W + w) * d.C + ts.c);
      }
      pw[i] += BK;
      while (pw[i] >= d.Q) {
        pw[i] -= d.Q;
        if (++ph[i] == d.P) { ph[i] = 0; ++nb[i]; }
      }
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int i = 0; i < NA; ++i) {
      const int mm = (tid + 256 * i) % BM, k = (tid + 256 * i) / BM;
      As[buf][k][mm] = d.op_bf16 ? rnd(DT_BF16, ra[i]) : ra[i];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float v = 0.f;
      if ((in >> i) & 1) {
        v = rb[i];
        if (d.x.scale) {
          v = fmaf(sc, v, sf);
          if (d.x.relu) v = fmaxf(v, 0.f);
        }
      }
      Bs[buf][pk + 4 * i][jn] = d.op_bf16 ? rnd(DT_BF16, v) : v;
    }
  };
  load(p_begin);
  store(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = p_begin; k0 < p_end; k0 += BK) {
    const bool more = k0 + BK < p_end;
    if (more) load(k0 + BK);
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      float a[TM], b[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = As[buf][k][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < TN; ++j) b[j] = Bs[buf][k][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    if (more) store(buf ^ 1);
    __syncthreads();
    buf ^= 1;
  }
  float* out = d.dw_part + (int64_t)split * d.K * RSC;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int ko = m0 + ty + 16 * i;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int jj = n0 + tx + 16 * j;
      if (ko < d.K && jj < RSC) out[(int64_t)ko * RSC + jj] = acc[i][j];
    }
  }
}

// Weight gradient of a conv with few input channels (the 3-channel stem and
// C^j convs): R*S*C <= 32 columns.  64-pixel steps stage dY and the im2col rows
// in shared memory; each of the eight warps takes every eighth pixel, its lanes
// hold the outputs -- KL = 16 or 32 output channels across the lanes, the
// columns of a pixel read as broadcast float4s -- so a pixel costs a lane one
// load of dY and one of every four columns.  The warps' sums meet in order at
// the end.  (One output a thread over all pixels of a step, two loads a
// multiply-add, took 819 us on the 64 x 64 stem of 256 images; now below 290.)
constexpr int kFewCols = 32;
template <int KL>
__global__ void __launch_bounds__(256) k_conv_wgrad_few(const ConvDesc* __restrict__ tab,
                                                        const int* __restrict__ tstart, int n) {
  constexpr int BM = kWgradBM, BP = 64, JG = 32 / KL;        // JG lane groups share the columns
  constexpr int KPL = KL == 16 ? 1 : BM / 32;                // output channels a lane
  constexpr int JV = kFewCols / 4 / JG;                      // float4 columns a lane
  __shared__ __align__(16) float As[BP][BM];                 // dY[pixel][k_out]; at the end the sums, as float4
  __shared__ __align__(16) float Bs[BP][kFewCols + 4];       // im2col[pixel][j]
  const int inst = find_instance(tstart, n, blockIdx.x);
  const ConvDesc d = tab[inst];
  int t = blockIdx.x - tstart[inst];
  const int tm = t % d.mtiles, split = t / d.mtiles;         // (one column tile)
  const int RSC = d.R * d.S * d.C, Mp = d.B * d.P * d.Q;
  const int m0 = tm * BM, km = min(BM, d.K - m0);
  const int p_begin = split * d.pix_per_split;
  const int p_end = min(Mp, p_begin + d.pix_per_split);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // staging: column j = lane
  const bool jin = lane < RSC;
  const TapStep ts(jin ? lane : 0, d.S, d.C);
  float sc = 1.f, sf = 0.f;
  if (d.x.scale) { sc = __ldg(d.x.scale + ts.c); sf = __ldg(d.x.shift + ts.c); }
  const int kl = lane % KL, jg = lane / KL;
  const int jv = (RSC + 3) / 4;                              // float4 columns in use
  float4 acc[KPL][JV];
#pragma unroll
  for (int a = 0; a < KPL; ++a)
#pragma unroll
    for (int v = 0; v < JV; ++v) acc[a][v] = make_float4(0.f, 0.f, 0.f, 0.f);
  // the next step's values wait in registers while a step is multiplied: dY
  // element tid + 256 i of the step's [64][km] block, column `lane` of pixels
  // warp + 8 i
  constexpr int ND = BP * BM / 256;
  float rd[KL == 16 ? ND / 4 : ND], rx[BP / 8];
  constexpr int NDK = KL == 16 ? ND / 4 : ND;
  int px = 0, py = 0, pi = 0;  // (column, row, image) of output pixel k0 + warp
  {
    const int pix = p_begin + warp;
    px = pix % d.Q;
    const int tmp = pix / d.Q;
    py = tmp % d.P;
    pi = tmp / d.P;
  }
  auto load = [&](int k0) {
    const int64_t row0 = (int64_t)k0 * d.K + m0;
#pragma unroll
    for (int i = 0; i < NDK; ++i) {
      const int e = tid + 256 * i, p = KL == 16 ? e >> 4 : e >> 6, k = KL == 16 ? e & 15 : e & 63;
      rd[i] = k < km && k0 + p < p_end ? __ldg(d.dy + row0 + (int64_t)p * d.K + k) : 0.f;
    }
#pragma unroll
    for (int i = 0; i < BP / 8; ++i) {
      const int h = py * d.stride - d.pad + ts.r, w = px * d.stride - d.pad + ts.s;
      float v = 0.f;
      if (jin && k0 + warp + 8 * i < p_end && h >= 0 && h < d.H && w >= 0 && w < d.W) {
        v = ldv(d.x.ptr, d.x.dt, ((int64_t)(pi * d.H + h) * d.W + w) * d.C + ts.c);
        if (d.x.scale) {
          v = fmaf(sc, v, sf);
          if (d.x.relu) v = fmaxf(v, 0.f);
        }
      }
      rx[i] = v;
      px += 8;
      while (px >= d.Q) {
        px -= d.Q;
        if (++py == d.P) { py = 0; ++pi; }
      }
    }
  };
  load(p_begin);
  for (int k0 = p_begin; k0 < p_end; k0 += BP) {
    __syncthreads();  // the previous step's tiles are consumed
#pragma unroll
    for (int i = 0; i < NDK; ++i) {
      const int e = tid + 256 * i, p = KL == 16 ? e >> 4 : e >> 6, k = KL == 16 ? e & 15 : e & 63;
      As[p][k] = d.op_bf16 ? rnd(DT_BF16, rd[i]) : rd[i];
    }
#pragma unroll
    for (int i = 0; i < BP / 8; ++i) Bs[warp + 8 * i][lane] = d.op_bf16 ? rnd(DT_BF16, rx[i]) : rx[i];
    __syncthreads();
    if (k0 + BP < p_end) load(k0 + BP);
#pragma unroll
    for (int i = 0; i < BP / 8; ++i) {
      const int px = warp + 8 * i;
      float a[KPL];
#pragma unroll
      for (int q = 0; q < KPL; ++q) a[q] = kl + 32 * q < km ? As[px][kl + 32 * q] : 0.f;
#pragma unroll
      for (int v = 0; v < JV; ++v) {
        const int col = v * JG + jg;
        if (v * JG >= jv) break;  // (columns past R*S*C are zero in Bs)
        const float4 b = *reinterpret_cast<const float4*>(&Bs[px][4 * col]);
#pragma unroll
        for (int q = 0; q < KPL; ++q) {
          acc[q][v].x = fmaf(a[q], b.x, acc[q][v].x);
          acc[q][v].y = fmaf(a[q], b.y, acc[q][v].y);
          acc[q][v].z = fmaf(a[q], b.z, acc[q][v].z);
          acc[q][v].w = fmaf(a[q], b.w, acc[q][v].w);
        }
      }
    }
  }
  // the eight warps' sums, one after another through shared memory
  float* sum = &As[0][0];  // [BM][kFewCols]
  for (int w = 0; w < 8; ++w) {
    __syncthreads();
    if (w != warp) continue;
#pragma unroll
    for (int q = 0; q < KPL; ++q)
#pragma unroll
      for (int v = 0; v < JV; ++v) {
        const int col = v * JG + jg, k = kl + 32 * q;
        float4* s4 = reinterpret_cast<float4*>(sum + k * kFewCols + 4 * col);
        float4 x = acc[q][v];
        if (w) {
          const float4 o = *s4;
          x = make_float4(o.x + x.x, o.y + x.y, o.z + x.z, o.w + x.w);
        }
        *s4 = x;
      }
  }
  __syncthreads();
  float* out = d.dw_part + (int64_t)split * d.K * RSC;
  for (int o = tid; o < km * RSC; o += 256) {
    const int k = o / RSC, j = o - k * RSC;
    out[(int64_t)(m0 + k) * RSC + j] = sum[k * kFewCols + j];
  }
}

// The same for 1x1 stride-1 convs (the C^j): at most 4 input channels, nothing
// to stage -- a warp takes every eighth pixel of the split, eight pixels' loads
// in flight, lanes across 64 output channels; the pixel's inputs are broadcast
// loads.  (The seven C^j of the 8-subnetwork ResNet-1001, batch 256: 443 -> 213 us.)
__global__ void __launch_bounds__(256) k_conv_wgrad_few1(const ConvDesc* __restrict__ tab,
                                                         const int* __restrict__ tstart, int n) {
  constexpr int BM = kWgradBM, U = 8, CM = 4;
  __shared__ float sum[8][BM][CM];
  const int inst = find_instance(tstart, n, blockIdx.x);
  const ConvDesc d = tab[inst];
  const int t = blockIdx.x - tstart[inst];
  const int tm = t % d.mtiles, split = t / d.mtiles;
  const int Mp = d.B * d.P * d.Q, m0 = tm * BM;
  const int p_begin = split * d.pix_per_split;
  const int p_end = min(Mp, p_begin + d.pix_per_split);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float sc[CM], sf[CM], acc[2][CM];
#pragma unroll
  for (int c = 0; c < CM; ++c) {
    sc[c] = d.x.scale && c < d.C ? __ldg(d.x.scale + c) : 1.f;
    sf[c] = d.x.scale && c < d.C ? __ldg(d.x.shift + c) : 0.f;
    acc[0][c] = acc[1][c] = 0.f;
  }
  const bool k0in = m0 + lane < d.K, k1in = m0 + 32 + lane < d.K;
  for (int p0 = p_begin + warp; p0 < p_end; p0 += 8 * U) {
    float dy[U][2], x[U][CM];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int p = p0 + 8 * u;
      const bool in = p < p_end;
      const float* g = d.dy + (int64_t)p * d.K + m0 + lane;
      dy[u][0] = in && k0in ? __ldg(g) : 0.f;
      dy[u][1] = in && k1in ? __ldg(g + 32) : 0.f;
#pragma unroll
      for (int c = 0; c < CM; ++c) x[u][c] = in && c < d.C ? ldv(d.x.ptr, d.x.dt, (int64_t)p * d.C + c) : 0.f;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (d.op_bf16) { dy[u][0] = rnd(DT_BF16, dy[u][0]); dy[u][1] = rnd(DT_BF16, dy[u][1]); }
#pragma unroll
      for (int c = 0; c < CM; ++c) {
        float v = x[u][c];
        if (d.x.scale) {
          v = fmaf(sc[c], v, sf[c]);  // (a pixel past the end has dY = 0)
          if (d.x.relu) v = fmaxf(v, 0.f);
        }
        if (d.op_bf16) v = rnd(DT_BF16, v);
        acc[0][c] = fmaf(dy[u][0], v, acc[0][c]);
        acc[1][c] = fmaf(dy[u][1], v, acc[1][c]);
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int c = 0; c < CM; ++c) sum[warp][lane + 32 * q][c] = acc[q][c];
  __syncthreads();
  float* out = d.dw_part + (int64_t)split * d.K * d.C;
  for (int o = threadIdx.x; o < BM * d.C; o += 256) {
    const int k = o / d.C, c = o - k * d.C;
    if (m0 + k >= d.K) continue;
    float v = sum[0][k][c];
#pragma unroll
    for (int w = 1; w < 8; ++w) v += sum[w][k][c];
    out[(int64_t)(m0 + k) * d.C + c] = v;
  }
}

// Forward conv with few input channels (R*S*C <= 32), 16 output channels a CTA
// row: one thread per output pixel loads its R*S*C inputs once and keeps the 16
// sums in registers, the weights broadcast from shared memory.  BN partials from
// the staged outputs, two passes over the CTA's 256 pixels.  (The tiled kernel
// took 290 us on the 64 x 64 stem of 256 images and 316 us on the C^j; both
// together now take 286.)
constexpr int kFewRows = 256;
__global__ void __launch_bounds__(256) k_conv_fwd_few(const ConvDesc* __restrict__ tab,
                                                      const int* __restrict__ tstart, int n) {
  constexpr int BN = 16;
  __shared__ __align__(16) float ws[kFewCols][BN];
  __shared__ int toff[kFewCols], tr[kFewCols], tsx[kFewCols];
  __shared__ float scs[kFewCols], sfs[kFewCols];
  __shared__ float st[kFewRows][BN + 1];
  const int inst = find_instance(tstart, n, blockIdx.x);
  const ConvDesc d = tab[inst];
  const int t = blockIdx.x - tstart[inst];
  const int tm = t % d.mtiles, tn = t / d.mtiles;
  const int M = d.B * d.P * d.Q, Kt = d.R * d.S * d.C;
  const int m0 = tm * kFewRows, n0 = tn * BN;
  const int tid = threadIdx.x;
  for (int e = tid; e < Kt * BN; e += 256) {
    const int k = e / BN, j = e % BN;
    ws[k][j] = n0 + j < d.K ? ldv(d.w, d.w_dt, (int64_t)(n0 + j) * Kt + k) : 0.f;
  }
  if (tid < Kt) {
    const TapStep ts(tid, d.S, d.C);
    tr[tid] = ts.r;
    tsx[tid] = ts.s;
    toff[tid] = (ts.r * d.W + ts.s) * d.C + ts.c;
    scs[tid] = d.x.scale ? __ldg(d.x.scale + ts.c) : 1.f;
    sfs[tid] = d.x.scale ? __ldg(d.x.shift + ts.c) : 0.f;
  }
  __syncthreads();
  const int m = m0 + tid;
  const bool mv = m < M;
  const int q = m % d.Q, tmp = m / d.Q, pp = tmp % d.P, nb = tmp / d.P;
  const int h0 = pp * d.stride - d.pad, w0 = q * d.stride - d.pad;
  const int64_t base = ((int64_t)(nb * d.H + h0) * d.W + w0) * d.C;
  float acc[BN];
#pragma unroll
  for (int j = 0; j < BN; ++j) acc[j] = 0.f;
  for (int k8 = 0; k8 < Kt; k8 += 8) {
    float v[8];
    unsigned in = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int k = k8 + e;
      v[e] = 0.f;
      if (k < Kt && mv) {
        const int h = h0 + tr[k], w = w0 + tsx[k];
        if (h >= 0 && h < d.H && w >= 0 && w < d.W) {
          in |= 1u << e;
          v[e] = ldv(d.x.ptr, d.x.dt, base + toff[k]);
        }
      }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int k = k8 + e;
      if (k >= Kt) break;
      float x = 0.f;
      if ((in >> e) & 1) {
        x = v[e];
        if (d.x.scale) {
          x = fmaf(scs[k], x, sfs[k]);
          if (d.x.relu) x = fmaxf(x, 0.f);
        }
      }
      if (d.op_bf16) x = rnd(DT_BF16, x);
#pragma unroll
      for (int j = 0; j < BN; j += 4) {
        const float4 w4 = *reinterpret_cast<const float4*>(&ws[k][j]);
        acc[j] = fmaf(x, w4.x, acc[j]);
        acc[j + 1] = fmaf(x, w4.y, acc[j + 1]);
        acc[j + 2] = fmaf(x, w4.z, acc[j + 2]);
        acc[j + 3] = fmaf(x, w4.w, acc[j + 3]);
      }
    }
  }
#pragma unroll
  for (int j = 0; j < BN; ++j) {
    const int co = n0 + j;
    if (!mv || co >= d.K) continue;
    const int64_t o = (int64_t)m * d.K + co;
    if (d.res) acc[j] += ldv(d.res, d.res_dt, o);
    if (d.res2[0]) acc[j] = fmaf(d.res2_c[0], ldv(d.res2[0], d.res2_dt[0], o), acc[j]);
    if (d.res2[1]) acc[j] = fmaf(d.res2_c[1], ldv(d.res2[1], d.res2_dt[1], o), acc[j]);
    acc[j] = rnd(d.y_dt, acc[j]);
  }
#pragma unroll
  for (int j = 0; j < BN; ++j) st[tid][j] = acc[j];
  __syncthreads();
  // stores with the channels of a pixel across neighbouring threads
  const int rows = min(kFewRows, M - m0);
  for (int e = tid; e < rows * BN; e += 256) {
    const int r = e / BN, j = e % BN;
    if (n0 + j < d.K) stv(d.y, d.y_dt, (int64_t)(m0 + r) * d.K + n0 + j, st[r][j]);
  }
  if (d.stats && d.stat_rows) {
    // partials of stat_rows rows in 16 row groups, as k_conv_fwd forms them
    __shared__ float2 red[16][BN];
    const int j = tid % BN, ty = tid / BN, tmr = d.stat_rows / 16;
    for (int r0 = 0; r0 < rows; r0 += d.stat_rows) {
      red[ty][j] = row_moments(tmr, m0 + r0 + ty, M, [&](int i) { return st[r0 + ty + 16 * i][j]; });
      __syncthreads();
      if (tid < BN && n0 + tid < d.K)
        merge_row_groups(tmr, m0 + r0, M, [&](int r) { return red[r][tid]; },
                         d.stats + ((int64_t)((m0 + r0) / d.stat_rows) * d.K + n0 + tid) * 2);
      __syncthreads();
    }
  } else if (d.stats) {
    // warp w: columns 2 w and 2 w + 1; lane l: rows l, l + 32, ...
    const int lane = tid & 31, warp = tid >> 5;
#pragma unroll
    for (int jj = 0; jj < 2; ++jj) {
      const int j = 2 * warp + jj;
      float s = 0.f;
      for (int r = lane; r < rows; r += 32) s += st[r][j];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      const float mean = s / (float)rows;
      float m2 = 0.f;
      for (int r = lane; r < rows; r += 32) m2 = fmaf(st[r][j] - mean, st[r][j] - mean, m2);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) m2 += __shfl_xor_sync(0xffffffffu, m2, o);
      if (lane == 0 && n0 + j < d.K) {
        d.stats[((int64_t)tm * d.K + n0 + j) * 2] = mean;
        d.stats[((int64_t)tm * d.K + n0 + j) * 2 + 1] = m2;
      }
    }
  }
}

// 128 consecutive partial positions per CTA, four a lane: warp w sums splits w,
// w+8, .. (512-byte rows of one split, four in flight), then the eight warp sums
// are added in warp order: a fixed order, so the result is deterministic.
// Transposed partials ([split][j][k_out]) land in dw[k_out][j].  (32 positions a
// CTA and one load in flight read 0.6 TB/s of VGG-16's partials: 876 us a step;
// now 380.)
__global__ void __launch_bounds__(256) k_wreduce(const WReduceDesc* __restrict__ tab, const int* __restrict__ tstart,
                                                 int n) {
  static_assert(kWreduceElems == 128, "four elements a lane");
  __shared__ float4 red[8][32];
  const int inst = find_instance(tstart, n, blockIdx.x);
  const WReduceDesc d = tab[inst];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t e0 = (int64_t)(blockIdx.x - tstart[inst]) * kWreduceElems + 4 * lane;
  const bool vec = (d.n & 3) == 0;
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  auto row = [&](int k) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    const float* p = d.part + (int64_t)k * d.n + e0;
    if (vec) {
      if (e0 < d.n) v = __ldg(reinterpret_cast<const float4*>(p));
    } else {
      if (e0 < d.n) v.x = __ldg(p);
      if (e0 + 1 < d.n) v.y = __ldg(p + 1);
      if (e0 + 2 < d.n) v.z = __ldg(p + 2);
      if (e0 + 3 < d.n) v.w = __ldg(p + 3);
    }
    return v;
  };
  auto add = [](float4& a, const float4& b) { a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w; };
  int k = w;
  for (; k + 24 < d.splits; k += 32) {
    const float4 v0 = row(k), v1 = row(k + 8), v2 = row(k + 16), v3 = row(k + 24);
    add(s, v0);
    add(s, v1);
    add(s, v2);
    add(s, v3);
  }
  for (; k < d.splits; k += 8) add(s, row(k));
  red[w][lane] = s;
  __syncthreads();
  // thread t < 128: element t of the CTA
  if (threadIdx.x >= kWreduceElems) return;
  const int64_t e = (int64_t)(blockIdx.x - tstart[inst]) * kWreduceElems + threadIdx.x;
  if (e >= d.n) return;
  const float* r = reinterpret_cast<const float*>(&red[0][0]) + threadIdx.x;
  float t = r[0];
#pragma unroll
  for (int i = 1; i < 8; ++i) t += r[i * kWreduceElems];
  const int64_t i = d.transposed ? (e % d.kout) * d.rsc + e / d.kout : e;
  d.dw[i] = d.accumulate ? d.dw[i] + t : t;
}

__global__ void k_wtrans(const WtDesc* __restrict__ tab, const int* __restrict__ tstart, int n) {
  const int inst = find_instance(tstart, n, blockIdx.x);
  const WtDesc& d = tab[inst];
  const int64_t i = (int64_t)(blockIdx.x - tstart[inst]) * blockDim.x + threadIdx.x;
  const uint16_t* src = reinterpret_cast<const uint16_t*>(d.src);
  if (d.pack == 0) {
    // one element a thread, in the order of the destination
    if (i >= d.n) return;
    const int k = (int)(i % d.K);
    const int64_t t = i / d.K;
    const int rs = (int)(t % d.RS), c = (int)(t / d.RS);
    reinterpret_cast<uint16_t*>(d.dst)[i] = src[((int64_t)k * d.RS + rs) * d.C + c];
    return;
  }
  // eight channels of one row and tap a thread: a 16-byte store; neighbouring
  // threads are neighbouring rows (pack 2: of consecutive addresses)
  if (8 * i >= d.n) return;
  const int all = d.pack == 1 ? d.K : d.C, rows = c3_block(all);
  const int64_t per = d.n / all * rows / 8;  // threads of a block of rows
  const int64_t j = i % per;
  const int row = (int)(i / per) * rows + (int)(j % rows);
  const int rs = (int)(j / rows % d.RS), ch = (int)(j / rows / d.RS) * 8;
  const int64_t step = d.pack == 1 ? 1 : (int64_t)d.RS * d.C;
  src += d.pack == 1 ? ((int64_t)row * d.RS + rs) * d.C + ch : ((int64_t)ch * d.RS + rs) * d.C + row;
  uint32_t w[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) w[e] = src[2 * e * step] | (uint32_t)src[(2 * e + 1) * step] << 16;
  reinterpret_cast<uint4*>(d.dst)[i] = make_uint4(w[0], w[1], w[2], w[3]);
}

// ---------------------------------------------------------------- row-tile geometry
// A tile is rows_per_tile rows x all C channels.  For C <= 256 (a power of
// two) thread t owns channel t % C and rows t / C + g * (256 / C); for
// C > 256 it owns channels t + 256 i and all rows.
struct RowTile {
  int G, cpt, c0, g;
  __device__ RowTile(int C, int tid) {
    if (C <= 256) {
      G = 256 / C; cpt = 1; c0 = tid % C; g = tid / C;
      if (g >= G) c0 = C;  // idle thread (C does not divide 256)
    } else { G = 1; cpt = (C + 255) / 256; c0 = tid; g = 0; }
  }
};

// A CTA takes a tile's rows of a slice of 64 channels (fewer: all), so that four
// or more threads share a channel's rows.  Rows are taken kEwBatch at a time, all
// loads of a batch first.  (All channels of the rows a CTA and one thread a
// channel left VGG-16's last interface, 512 x 512, eight CTAs with a chain of 64
// rows: 98 us,
// 91 with the batches; 36 now, of which an event-timed launch is about 8.)
constexpr int kEwBatch = 8;
__global__ void __launch_bounds__(256) k_ew(const EwDesc* __restrict__ tab, const int* __restrict__ tstart, int n) {
  __shared__ float red[256][2];
  const int inst = find_instance(tstart, n, blockIdx.x);
  const EwDesc& d = tab[inst];
  const int C = d.C;
  int tile = blockIdx.x - tstart[inst], cb = 0;
  if (C > kEwSlice) {
    const int slices = ew_slices(C), item = tile;
    tile = item / slices;
    cb = (item - tile * slices) * kEwSlice;
  }
  const int Cs = min(C - cb, kEwSlice);
  const int G = d.groups ? d.groups : 256 / Cs;                  // row groups
  const int g = threadIdx.x / Cs, c = cb + threadIdx.x % Cs;     // (g >= G: an idle thread)
  const int64_t r0 = (int64_t)tile * d.rows_per_tile;
  const int64_t r1 = min((int64_t)d.M, r0 + d.rows_per_tile);
  // BN partials of the output: Welford's update over this thread's rows
  // (count, mean, M2), then chan_merge over the row groups in order
  float cnt = 0.f, mean = 0.f, m2 = 0.f;
  if (g < G) {
    for (int64_t r = r0 + g; r < r1; r += (int64_t)kEwBatch * G) {
      float v[kEwBatch];
#pragma unroll
      for (int u = 0; u < kEwBatch; ++u) v[u] = 0.f;
      for (int i = 0; i < d.nin; ++i) {
        const Src src = d.in[i];
        float x[kEwBatch];
#pragma unroll
        for (int u = 0; u < kEwBatch; ++u) {
          const int64_t rr = r + (int64_t)u * G;
          x[u] = rr < r1 ? ld_src(src, rr * C + c, c) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < kEwBatch; ++u) v[u] = fmaf(d.coef[i], x[u], v[u]);
      }
#pragma unroll
      for (int u = 0; u < kEwBatch; ++u) {
        const int64_t rr = r + (int64_t)u * G;
        if (rr >= r1) break;
        float y = v[u];
        if (d.relu) y = fmaxf(y, 0.f);
        if (d.out) {
          y = rnd(d.out_dt, y);
          stv(d.out, d.out_dt, rr * C + c, y);
        }
        if (d.stats) {
          cnt += 1.f;
          const float delta = y - mean;
          mean += delta / cnt;
          m2 = fmaf(delta, y - mean, m2);
        }
      }
    }
  }
  if (d.stats) {
    red[threadIdx.x][0] = mean;
    red[threadIdx.x][1] = m2;
    __syncthreads();
    if ((int)threadIdx.x < Cs) {
      float a = 0.f, am = 0.f, a2 = 0.f;
      for (int q = 0; q < G; ++q) {
        // rows r0 + q, r0 + q + G, ... below r1
        const float cq = r1 > r0 + q ? (float)((r1 - r0 - q + G - 1) / G) : 0.f;
        chan_merge(a, am, a2, cq, red[q * Cs + threadIdx.x][0], red[q * Cs + threadIdx.x][1]);
      }
      float* out = d.stats + ((int64_t)tile * C + cb + threadIdx.x) * 2;
      out[0] = am;
      out[1] = a2;
    }
  }
}

__global__ void __launch_bounds__(256) k_ew_bwd(const EwBwdDesc* __restrict__ tab, const int* __restrict__ tstart,
                                                int n) {
  constexpr int U = 4;  // elements a thread has in flight
  const int inst = find_instance(tstart, n, blockIdx.x);
  const EwBwdDesc& d = tab[inst];
  const int tile = blockIdx.x - tstart[inst];
  const int elems = ew_bwd_elems(d.C);
  const int64_t base = (int64_t)tile * elems;
  const int64_t end = min((int64_t)d.M * d.C, base + elems);
  for (int64_t o = base + threadIdx.x; o < end; o += U * 256) {
    float g[U];
#pragma unroll
    for (int u = 0; u < U; ++u) g[u] = o + 256 * u < end ? d.dout[o + 256 * u] : 0.f;
    if (d.relu) {
      float y[U];
#pragma unroll
      for (int u = 0; u < U; ++u) y[u] = o + 256 * u < end ? ldv(d.out, d.out_dt, o + 256 * u) : 0.f;
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (!(y[u] > 0.f)) g[u] = 0.f;
    }
    for (int i = 0; i < d.nin; ++i) {
      float* gin = d.gin[i];
      float a[U];
#pragma unroll
      for (int u = 0; u < U; ++u) a[u] = d.acc[i] && o + 256 * u < end ? gin[o + 256 * u] : 0.f;
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (o + 256 * u < end) {
          const float v = d.coef[i] * g[u];
          gin[o + 256 * u] = d.acc[i] ? a[u] + v : v;
        }
    }
  }
}

// ---------------------------------------------------------------- BN
// Finalisation of the per-tile BN partials ([tiles][C][2] floats, a few MB at
// most): latency bounds it, so one CTA takes 8 channels and all their tiles in
// a single level -- thread = (channel t & 7, tile lane t >> 3), 64 tile lanes,
// 16 loads in flight a thread, one pass through shared memory.  There is no
// second level (the former 32 channels x 64 tiles a CTA met in global scratch
// behind an atomic count: five dependent trips to L2).  Sums run as unevaluated
// sums of floats (Knuth's TwoSum) -- two, about 48 bits, for the forward's fp32
// terms; three, more than the 53 bits of fp64, for the backward's -- since this
// part's fp64 pipe would take longer than the loads.  The training step of the
// 8-subnetwork ResNet-1001 (batch 256, 64 px; 340 such launches of up to 2048
// tiles a layer): 81.94 -> 81.36 ms with two floats, one quantity at a time.  Both
// quantities of a partial packed, with the third float: 4-subnetwork ResNet-1001
// (batch 128, 32 px) 26.27 -> 26.01 ms a step; unpacked, the third float had cost 0.17 ms, and
// with 4 channels a CTA 0.5 ms.
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
  return tc::fma2(b, tc::pk2(-1.f, -1.f), a);  // (one rounding: a - b)
}
// a + b -> its fp32 rounding, e: what that leaves out
__device__ __forceinline__ uint64_t two_sum(uint64_t a, uint64_t b, uint64_t& e) {
  const uint64_t s = tc::add2(a, b), bb = sub2(s, a);
  e = tc::add2(sub2(a, sub2(s, bb)), sub2(b, bb));
  return s;
}
template <int N>
struct FloatSum {
  uint64_t v[N] = {};  // decreasing
  // x into part `from` and its remainders into the following ones
  __device__ __forceinline__ void add(uint64_t x, int from = 0) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      if (i < from) continue;
      if (i == N - 1) v[i] = tc::add2(v[i], x);
      else v[i] = two_sum(v[i], x, x);
    }
  }
  __device__ __forceinline__ void add(const FloatSum& o) {
#pragma unroll
    for (int i = 0; i < N; ++i) add(o.v[i], i);
  }
  // as two floats: nothing cancels any more, and 48 bits are to become an fp32
  // (an overflowed or NaN sum is its first part)
  __device__ __forceinline__ void pair(uint64_t& hi, uint64_t& lo) const {
    hi = v[0];
    lo = v[1];
    if (N == 2) return;
    hi = two_sum(v[0], v[1], lo);
    lo = tc::add2(lo, v[N - 1]);
    hi = two_sum(hi, lo, lo);
    const float2 a = tc::un2(v[0]), b = tc::un2(hi);
    hi = tc::pk2(isfinite(a.x) ? b.x : a.x, isfinite(a.y) ? b.y : a.y);
  }
};
// (an overflowed or NaN sum has no meaningful low part)
__device__ __forceinline__ double pair_value(float hi, float lo) {
  return isfinite(hi) ? (double)hi + (double)lo : (double)hi;
}

constexpr int kFinThreads = 512;
constexpr int kFinLanes = kFinThreads / kFinChannels;  // tile lanes
constexpr int kFinUnroll = 16;                         // loads in flight a thread

// Sums over all tiles for the 8 channels of group cg.  MOMENTS false: of the
// two partial quantities.  MOMENTS true: the tiles hold (mean_t, M2_t) of
// n_t rows (rpt rows each, the last tile the remainder of M), combined as
// shifted sums around K = mean_0 (the first tile's mean): with d_t = mean_t - K,
//   S1 = sum n_t d_t,   S2 = sum (M2_t + n_t d_t^2),
//   mean = K + S1 / M,  M2 = S2 - S1^2 / M,
// which is Chan's pairwise update written for many sets at once (no term
// subtracts two large sums: K lies within a few standard errors of the mean,
// so S1^2 / M is a small part of S2).  Fixed order; threads 0 .. 7 return the
// sums of their channel.
template <bool MOMENTS>
__device__ __forceinline__ void tile_sums(const float* __restrict__ part, int C, int tiles, int64_t M, int rpt, int cg,
                                          double& s1, double& s2, float& K) {
  constexpr int N = MOMENTS ? 2 : 3;
  using Sum = FloatSum<N>;
  __shared__ uint64_t red[N][kFinLanes][kFinChannels + 1];
  __shared__ uint64_t tot[kFinChannels][2];
  const int ch = threadIdx.x % kFinChannels, tl = threadIdx.x / kFinChannels;
  const int c = cg * kFinChannels + ch;
  Sum a;
  K = 0.f;
  if (c < C) {
    const float2* p = reinterpret_cast<const float2*>(part) + c;
    if (MOMENTS && tiles > 0) K = __ldg(part + (int64_t)c * 2);
    const float full = (float)rpt, last = (float)(M - (int64_t)(tiles - 1) * rpt);  // rows of a tile
    for (int t0 = tl; t0 < tiles; t0 += kFinLanes * kFinUnroll) {
      float2 v[kFinUnroll];
#pragma unroll
      for (int k = 0; k < kFinUnroll; ++k) {
        const int t = t0 + k * kFinLanes;
        v[k] = t < tiles ? __ldg(p + (int64_t)t * C) : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int k = 0; k < kFinUnroll; ++k) {
        const int t = t0 + k * kFinLanes;
        if (t >= tiles) continue;
        if (MOMENTS) {
          const float n = t + 1 < tiles ? full : last;
          const float d = v[k].x - K;
          const float nd = n * d;
          a.add(tc::pk2(nd, fmaf(nd, d, v[k].y)));
        } else {
          a.add(tc::pk2(v[k].x, v[k].y));
        }
      }
    }
  }
#pragma unroll
  for (int i = 0; i < N; ++i) red[i][tl][ch] = a.v[i];
  __syncthreads();
  if (const int w = threadIdx.x >> 5, lane = threadIdx.x & 31; w < kFinChannels) {
    Sum s;
#pragma unroll
    for (int i = 0; i < N; ++i) s.v[i] = red[i][lane][w];
#pragma unroll
    for (int l = 32; l < kFinLanes; l += 32) {
      if (l >= tiles) break;  // (a lane without a tile holds zero)
      Sum o;
#pragma unroll
      for (int i = 0; i < N; ++i) o.v[i] = red[i][lane + l][w];
      s.add(o);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      if (o >= tiles) continue;
      Sum t;
#pragma unroll
      for (int i = 0; i < N; ++i) t.v[i] = __shfl_xor_sync(0xffffffffu, s.v[i], o);
      s.add(t);
    }
    if (lane == 0) s.pair(tot[w][0], tot[w][1]);
  }
  __syncthreads();
  s1 = s2 = 0.0;
  if (threadIdx.x < kFinChannels) {
    const float2 h = tc::un2(tot[threadIdx.x][0]), l = tc::un2(tot[threadIdx.x][1]);
    s1 = pair_value(h.x, l.x);
    s2 = pair_value(h.y, l.y);
  }
}

// The moments in the fixed order of an fp32 network (see the top): eight tiles of a
// chunk of 64, w + 8 k, in fp32; the chunk's eight sums in order; the chunks w,
// w + 8, ... and then the eight sums of chunks, all in fp64.  Tile lane l of a CTA is
// sum l & 7 of chunk l >> 3 of the 512 tiles of a round.
__device__ __forceinline__ void tile_moments_fixed(const float* __restrict__ part, int C, int tiles, int64_t M, int rpt,
                                                   int cg, double& s1, double& s2, float& K) {
  constexpr int Q = 2 * kFinChannels;
  __shared__ double red[kFinLanes][Q + 1];
  __shared__ double tot[8][Q];
  const int tid = threadIdx.x, ch = tid % kFinChannels, l = tid / kFinChannels;
  const int c = cg * kFinChannels + ch;
  K = c < C && tiles > 0 ? __ldg(part + (int64_t)c * 2) : 0.f;
  double acc = 0.0;  // thread 16 j + q: quantity q of the chunks j, j + 8, ...
  for (int t0 = 0; t0 < tiles; t0 += 8 * kFinLanes) {
    const int b = t0 + (l >> 3) * 64 + (l & 7);
    float2 v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k)
      v[k] = c < C && b + 8 * k < tiles ? __ldg(reinterpret_cast<const float2*>(part) + (int64_t)(b + 8 * k) * C + c)
                                        : make_float2(0.f, 0.f);
    float fa = 0.f, fb = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int64_t t = b + 8 * k;
      if (t < tiles) {
        const int64_t r1 = (t + 1) * rpt < M ? (t + 1) * rpt : M;
        const float n = (float)(r1 - t * rpt);
        const float d = v[k].x - K;
        const float nd = n * d;
        fa += nd;
        fb += v[k].y + nd * d;
      }
    }
    red[l][2 * ch] = fa;
    red[l][2 * ch + 1] = fb;
    __syncthreads();
    if (tid < 8 * Q) {
      double s = 0.0;
#pragma unroll
      for (int w = 0; w < 8; ++w) s += red[tid / Q * 8 + w][tid % Q];
      acc += s;
    }
    __syncthreads();
  }
  if (tid < 8 * Q) tot[tid / Q][tid % Q] = acc;
  __syncthreads();
  s1 = s2 = 0.0;
  if (tid < kFinChannels)
    for (int j = 0; j < 8; ++j) {
      s1 += tot[j][2 * tid];
      s2 += tot[j][2 * tid + 1];
    }
}

// scale and shift of a BN layer from the statistics it normalises with
__device__ __forceinline__ void bn_affine(const BnFinDesc& d, int c, float gamma, float beta, float mean, float var) {
  const float rstd = 1.f / sqrtf(var + 1e-5f);
  const float sc = gamma * rstd;
  d.mean[c] = mean;
  d.rstd[c] = rstd;
  d.scale[c] = sc;
  d.shift[c] = fmaf(-mean, sc, beta);
}

template <bool FIXED>
__global__ void __launch_bounds__(kFinThreads) k_bn_fin(const BnFinDesc* __restrict__ tab,
                                                        const int* __restrict__ tstart, int n) {
  const int inst = find_instance(tstart, n, blockIdx.x);
  const BnFinDesc d = tab[inst];
  const int cg = blockIdx.x - tstart[inst];
  const int c = cg * kFinChannels + threadIdx.x;
  const bool fin = threadIdx.x < kFinChannels && c < d.C;
  // the layer's parameters, loaded beside the partials
  float gamma = 0.f, beta = 0.f, rm = 0.f, rv = 0.f;
  if (fin) {
    gamma = d.gamma[c];
    beta = d.beta[c];
    if (d.run_mean) { rm = d.run_mean[c]; rv = d.run_var[c]; }
  }
  double s1, s2;
  float K;
  if (FIXED) tile_moments_fixed(d.part, d.C, d.tiles, d.count, d.rows_per_tile, cg, s1, s2, K);
  else tile_sums<true>(d.part, d.C, d.tiles, d.count, d.rows_per_tile, cg, s1, s2, K);
  if (!fin) return;
  // (1 / count comes from the host: no fp64 division here; from the moments on
  // fp32 holds every quantity to 2^-24)
  const float mean = (float)((double)K + s1 * d.inv_count);
  const float m2 = (float)(s2 - s1 * s1 * d.inv_count);
  float var = d.count > 0 ? m2 / (float)d.count : 0.f;
  if (var < 0.f) var = 0.f;
  if (d.run_mean) {
    // running statistics follow the batch mean and the unbiased variance
    const float m = d.momentum;
    const float unbiased = d.count > 1 ? var * ((float)d.count / (float)(d.count - 1)) : var;
    d.run_mean[c] = fmaf(m, mean, (1.f - m) * rm);
    d.run_var[c] = fmaf(m, unbiased, (1.f - m) * rv);
  }
  bn_affine(d, c, gamma, beta, mean, var);
}

// eval mode: the running statistics stand in for the batch's (one thread per channel)
__global__ void __launch_bounds__(kFinEvalChannels) k_bn_eval(const BnFinDesc* __restrict__ tab,
                                                              const int* __restrict__ tstart, int n) {
  const int inst = find_instance(tstart, n, blockIdx.x);
  const BnFinDesc& d = tab[inst];
  const int c = (blockIdx.x - tstart[inst]) * kFinEvalChannels + threadIdx.x;
  if (c < d.C) bn_affine(d, c, d.gamma[c], d.beta[c], d.run_mean[c], d.run_var[c]);
}

__global__ void __launch_bounds__(256) k_bnb_reduce(const BnBwdDesc* __restrict__ tab,
                                                    const int* __restrict__ tstart, int n) {
  __shared__ float red[256][2];
  const int inst = find_instance(tstart, n, blockIdx.x);
  const BnBwdDesc& d = tab[inst];
  const int tile = blockIdx.x - tstart[inst];
  const int C = d.C;
  const RowTile rt(C, threadIdx.x);
  const int64_t r0 = (int64_t)tile * d.rows_per_tile;
  const int64_t r1 = min((int64_t)d.M, r0 + d.rows_per_tile);
  for (int ci = 0; ci < rt.cpt; ++ci) {
    const int c = rt.c0 + 256 * ci;
    float s1 = 0.f, s2 = 0.f;
    if (c < C) {
      const float mean = d.mean[c], rstd = d.rstd[c], sc = d.scale[c], sh = d.shift[c];
      for (int64_t r = r0 + rt.g; r < r1; r += rt.G) {
        const int64_t o = r * C + c;
        const float h = ldv(d.h, d.h_dt, o);
        float dz = d.da[o];
        if (d.relu && !(fmaf(sc, h, sh) > 0.f)) dz = 0.f;
        s1 += dz;
        s2 += dz * ((h - mean) * rstd);
      }
    }
    if (rt.G == 1) {
      if (c < C) {
        d.part[((int64_t)tile * C + c) * 2] = s1;
        d.part[((int64_t)tile * C + c) * 2 + 1] = s2;
      }
    } else {
      red[threadIdx.x][0] = s1;
      red[threadIdx.x][1] = s2;
      __syncthreads();
      if ((int)threadIdx.x < C) {
        float a = 0.f, b = 0.f;
        for (int g = 0; g < rt.G; ++g) { a += red[g * C + threadIdx.x][0]; b += red[g * C + threadIdx.x][1]; }
        d.part[((int64_t)tile * C + threadIdx.x) * 2] = a;
        d.part[((int64_t)tile * C + threadIdx.x) * 2 + 1] = b;
      }
      __syncthreads();
    }
  }
}

__global__ void __launch_bounds__(kFinThreads) k_bnb_fin(const BnBwdDesc* __restrict__ tab,
                                                         const int* __restrict__ tstart, int n) {
  const int inst = find_instance(tstart, n, blockIdx.x);
  const BnBwdDesc d = tab[inst];
  const int cg = blockIdx.x - tstart[inst];
  const int c = cg * kFinChannels + threadIdx.x;
  const bool fin = threadIdx.x < kFinChannels && c < d.C;
  float k0 = 0.f, b0 = 0.f, g0 = 0.f;
  if (fin) {
    k0 = d.gamma[c] * d.rstd[c];
    if (d.accumulate) { b0 = d.dbeta[c]; g0 = d.dgamma[c]; }
  }
  double s1, s2;
  float unused;
  tile_sums<false>(d.part, d.C, d.tiles, d.M, 0, cg, s1, s2, unused);
  if (!fin) return;
  d.dbeta[c] = d.accumulate ? b0 + (float)s1 : (float)s1;
  d.dgamma[c] = d.accumulate ? g0 + (float)s2 : (float)s2;
  d.coef[c * 3 + 0] = k0;
  d.coef[c * 3 + 1] = (float)(s1 * d.inv_count);
  d.coef[c * 3 + 2] = (float)(s2 * d.inv_count);
}

__global__ void __launch_bounds__(256) k_bnb_apply(const BnBwdDesc* __restrict__ tab,
                                                   const int* __restrict__ tstart, int n) {
  const int inst = find_instance(tstart, n, blockIdx.x);
  const BnBwdDesc& d = tab[inst];
  const int tile = blockIdx.x - tstart[inst];
  const int C = d.C;
  const int64_t base = (int64_t)tile * d.rows_per_tile * C;
  const int64_t end = min((int64_t)d.M * C, base + (int64_t)d.rows_per_tile * C);
  for (int64_t o = base + threadIdx.x; o < end; o += blockDim.x) {
    const int c = (int)(o % C);
    const float h = ldv(d.h, d.h_dt, o);
    float dz = d.da[o];
    if (d.relu && !(fmaf(d.scale[c], h, d.shift[c]) > 0.f)) dz = 0.f;
    const float xhat = (h - d.mean[c]) * d.rstd[c];
    float v = d.coef[c * 3] * (dz - d.coef[c * 3 + 1] - xhat * d.coef[c * 3 + 2]);
    if (d.add0) v = fmaf(d.add_c[0], d.add0[o], v);
    if (d.add1) v = fmaf(d.add_c[1], d.add1[o], v);
    d.dh[o] = d.accumulate ? d.dh[o] + v : v;
  }
}

// ---------------------------------------------------------------- BN backward, 8 channels per thread
// Used when C % 8 == 0: each thread moves 8 consecutive channels of one row
// with 16/32-byte accesses.
__device__ __forceinline__ void ld8f(const float* p, float* v) {
  const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void st8f(float* p, const float* v) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  *reinterpret_cast<float4*>(p + 4) = make_float4(v[4], v[5], v[6], v[7]);
}
__device__ __forceinline__ void ld8any(const void* base, int dt, int64_t i, float* v) {
  if (dt == DT_F32) {
    ld8f(reinterpret_cast<const float*>(base) + i, v);
  } else {
    const uint4 u = *reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(base) + i);
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2 f = __bfloat1622float2(h[k]);
      v[2 * k] = f.x;
      v[2 * k + 1] = f.y;
    }
  }
}

__global__ void __launch_bounds__(256) k_bnb_reduce8(const BnBwdDesc* __restrict__ tab,
                                                     const int* __restrict__ tstart, int n) {
  __shared__ float red[16][256];  // [quantity x channel][thread]: a warp touches 32 consecutive words
  const int inst = find_instance(tstart, n, blockIdx.x);
  const BnBwdDesc d = tab[inst];
  const int tile = blockIdx.x - tstart[inst];
  const int C = d.C, CG = C / 8;
  const int G = 256 / CG;  // row groups (CG <= 256)
  const int cg = threadIdx.x % CG, g = threadIdx.x / CG;
  const int64_t r0 = (int64_t)tile * d.rows_per_tile;
  const int64_t r1 = min((int64_t)d.M, r0 + d.rows_per_tile);
  float s1[8], s2[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) { s1[k] = 0.f; s2[k] = 0.f; }
  if (g < G) {
    const int c0 = cg * 8;
    float mean[8], rstd[8], sc[8], sh[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      mean[k] = d.mean[c0 + k]; rstd[k] = d.rstd[c0 + k]; sc[k] = d.scale[c0 + k]; sh[k] = d.shift[c0 + k];
    }
    for (int64_t r = r0 + g; r < r1; r += G) {
      const int64_t o = r * C + c0;
      float h[8], dz[8];
      ld8any(d.h, d.h_dt, o, h);
      ld8f(d.da + o, dz);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        if (d.relu && !(fmaf(sc[k], h[k], sh[k]) > 0.f)) dz[k] = 0.f;
        s1[k] += dz[k];
        s2[k] += dz[k] * ((h[k] - mean[k]) * rstd[k]);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 8; ++k) { red[k][threadIdx.x] = s1[k]; red[8 + k][threadIdx.x] = s2[k]; }
  __syncthreads();
  int groups = G;
  if ((G & (G - 1)) == 0) {
    // tree over the row groups: red[.][g * CG + cg] += red[.][(g + st) * CG + cg]
    for (int st = G >> 1; st > 0; st >>= 1) {
      if (g < st) {
#pragma unroll
        for (int k = 0; k < 16; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + st * CG];
      }
      __syncthreads();
    }
    groups = 1;
  }
  if ((int)threadIdx.x < CG) {
    float a[8], b[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) { a[k] = 0.f; b[k] = 0.f; }
    for (int gg = 0; gg < groups; ++gg)
#pragma unroll
      for (int k = 0; k < 8; ++k) { a[k] += red[k][gg * CG + threadIdx.x]; b[k] += red[8 + k][gg * CG + threadIdx.x]; }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      d.part[((int64_t)tile * C + threadIdx.x * 8 + k) * 2] = a[k];
      d.part[((int64_t)tile * C + threadIdx.x * 8 + k) * 2 + 1] = b[k];
    }
  }
}

// The same sums for an fp32 network, in the fixed order: the tall tiles of
// bnb_fixed_rows, G = 256 / (C / 8) row groups one row after another, the groups in
// k_bnb_reduce8's tree.  A CTA takes half of a tile's channels, a thread four of them
// with all its rows in flight (16 a thread up to 128 channels).  (8 channels a thread,
// eight rows in flight, one CTA a tile: 10.4 us a launch of the tiny network under
// ncu, now 8.1; its step 255 -> 251 us.)
__global__ void __launch_bounds__(256) k_bnb_reduce_fixed(const BnBwdDesc* __restrict__ tab,
                                                          const int* __restrict__ tstart, int n) {
  constexpr int U = 16;
  __shared__ float red[8][256];
  const int inst = find_instance(tstart, n, blockIdx.x);
  const BnBwdDesc d = tab[inst];
  const int t = blockIdx.x - tstart[inst], tile = t >> 1;
  const int C = d.C, CG = C / 8, G = 256 / CG;  // CG quads of channels a CTA
  const int q = threadIdx.x % CG, g = threadIdx.x / CG, c0 = ((t & 1) * CG + q) * 4;
  const int64_t r0 = (int64_t)tile * d.rows_per_tile;
  const int64_t r1 = min((int64_t)d.M, r0 + d.rows_per_tile);
  const float* hp = static_cast<const float*>(d.h);
  float s1[4] = {}, s2[4] = {};
  if (g < G) {
    float mean[4], rstd[4], sc[4], sh[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      mean[k] = d.mean[c0 + k]; rstd[k] = d.rstd[c0 + k]; sc[k] = d.scale[c0 + k]; sh[k] = d.shift[c0 + k];
    }
    for (int64_t r = r0 + g; r < r1; r += U * G) {
      float4 hv[U], dv[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (r + u * G >= r1) break;
        const int64_t o = (r + u * G) * C + c0;
        hv[u] = *reinterpret_cast<const float4*>(hp + o);
        dv[u] = *reinterpret_cast<const float4*>(d.da + o);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (r + u * G >= r1) break;
        const float h[4] = {hv[u].x, hv[u].y, hv[u].z, hv[u].w};
        float dz[4] = {dv[u].x, dv[u].y, dv[u].z, dv[u].w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (d.relu && !(fmaf(sc[k], h[k], sh[k]) > 0.f)) dz[k] = 0.f;
          s1[k] += dz[k];
          s2[k] += dz[k] * ((h[k] - mean[k]) * rstd[k]);
        }
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) { red[k][threadIdx.x] = s1[k]; red[4 + k][threadIdx.x] = s2[k]; }
  __syncthreads();
  int groups = G;
  if ((G & (G - 1)) == 0) {
    for (int st = G >> 1; st > 0; st >>= 1) {
      if (g < st) {
#pragma unroll
        for (int k = 0; k < 8; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + st * CG];
      }
      __syncthreads();
    }
    groups = 1;
  }
  if ((int)threadIdx.x < CG) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float a = 0.f, b = 0.f;
      for (int gg = 0; gg < groups; ++gg) {
        a += red[k][gg * CG + q];
        b += red[4 + k][gg * CG + q];
      }
      reinterpret_cast<float2*>(d.part)[(int64_t)tile * C + c0 + k] = make_float2(a, b);
    }
  }
}

// Each thread keeps one group of 8 channels (cg = thread % (C/8)) for the
// whole tile, with that group's per-channel parameters in registers, and
// walks the tile's rows G = 256 / (C/8) apart.
__global__ void __launch_bounds__(256) k_bnb_apply8(const BnBwdDesc* __restrict__ tab,
                                                    const int* __restrict__ tstart, int n) {
  const int inst = find_instance(tstart, n, blockIdx.x);
  const BnBwdDesc d = tab[inst];  // a private copy: the stores below cannot force reloads
  const int tile = blockIdx.x - tstart[inst];
  const int C = d.C, CG = C / 8;
  const int G = 256 / CG;
  const int cg = threadIdx.x % CG, g = threadIdx.x / CG;
  if (g >= G) return;
  const int c0 = cg * 8;
  float sc[8], sh[8], mean[8], rstd[8], k0[8], k1[8], k2[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    sc[k] = d.scale[c0 + k]; sh[k] = d.shift[c0 + k]; mean[k] = d.mean[c0 + k]; rstd[k] = d.rstd[c0 + k];
    k0[k] = d.coef[(c0 + k) * 3]; k1[k] = d.coef[(c0 + k) * 3 + 1]; k2[k] = d.coef[(c0 + k) * 3 + 2];
  }
  const int64_t r0 = (int64_t)tile * d.rows_per_tile;
  const int64_t r1 = min((int64_t)d.M, r0 + d.rows_per_tile);
  for (int64_t r = r0 + g; r < r1; r += G) {
    const int64_t o = r * C + c0;
    float h[8], dz[8], out[8];
    ld8any(d.h, d.h_dt, o, h);
    ld8f(d.da + o, dz);
    float a0[8], a1[8], ac[8];
    if (d.add0) ld8f(d.add0 + o, a0);
    if (d.add1) ld8f(d.add1 + o, a1);
    if (d.accumulate) ld8f(d.dh + o, ac);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (d.relu && !(fmaf(sc[k], h[k], sh[k]) > 0.f)) dz[k] = 0.f;
      const float xhat = (h[k] - mean[k]) * rstd[k];
      out[k] = k0[k] * (dz[k] - k1[k] - xhat * k2[k]);
      if (d.add0) out[k] = fmaf(d.add_c[0], a0[k], out[k]);
      if (d.add1) out[k] = fmaf(d.add_c[1], a1[k], out[k]);
      if (d.accumulate) out[k] += ac[k];
    }
    st8f(d.dh + o, out);
  }
}

// ---------------------------------------------------------------- pooling
// A thread takes V = 4 consecutive channels of a pixel where C allows it (the
// index arithmetic is once a thread, the loads 8 or 16 bytes), else one.
template <int V>
struct PoolSrc {
  const PoolDesc& d;
  int c;
  float sc[V], sf[V];
  __device__ __forceinline__ PoolSrc(const PoolDesc& desc, int ch) : d(desc), c(ch) {
    if (d.x.scale)
#pragma unroll
      for (int i = 0; i < V; ++i) { sc[i] = __ldg(d.x.scale + c + i); sf[i] = __ldg(d.x.shift + c + i); }
  }
  __device__ __forceinline__ void get(int64_t pix, float* v) const {
    const int64_t o = pix * d.C + c;
    if (V == 4 && d.x.dt == DT_BF16) {
      const uint2 u = __ldg(reinterpret_cast<const uint2*>(reinterpret_cast<const __nv_bfloat16*>(d.x.ptr) + o));
      const uint32_t w[2] = {u.x, u.y};
#pragma unroll
      for (int i = 0; i < V; ++i) v[i] = __uint_as_float((i & 1) ? w[i >> 1] & 0xffff0000u : w[i >> 1] << 16);
    } else if (V == 4) {
      const float4 f = __ldg(reinterpret_cast<const float4*>(reinterpret_cast<const float*>(d.x.ptr) + o));
      const float q[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
      for (int i = 0; i < V; ++i) v[i] = q[i];
    } else {
      v[0] = ldv(d.x.ptr, d.x.dt, o);
    }
    if (d.x.scale) {
#pragma unroll
      for (int i = 0; i < V; ++i) {
        v[i] = fmaf(sc[i], v[i], sf[i]);
        if (d.x.relu) v[i] = fmaxf(v[i], 0.f);
      }
    }
  }
};

template <int V>
__device__ __forceinline__ void pool_fwd_at(const PoolDesc& d, int64_t i) {
  const int c = (int)(i % d.C);
  int64_t t = i / d.C;
  const int q = (int)(t % d.Q); t /= d.Q;
  const int p = (int)(t % d.P);
  const int nb = (int)(t / d.P);
  const PoolSrc<V> src(d, c);
  float best[V];
#pragma unroll
  for (int j = 0; j < V; ++j) best[j] = -INFINITY;
  for (int r = 0; r < d.k; ++r)
    for (int s = 0; s < d.k; ++s) {
      const int h = p * d.stride + r - d.pad, w = q * d.stride + s - d.pad;
      if (h < 0 || h >= d.H || w < 0 || w >= d.W) continue;
      float v[V];
      src.get((int64_t)(nb * d.H + h) * d.W + w, v);
#pragma unroll
      for (int j = 0; j < V; ++j)
        if (v[j] > best[j]) best[j] = v[j];
    }
#pragma unroll
  for (int j = 0; j < V; ++j) stv(d.y, d.y_dt, i + j, best[j]);
}
__global__ void __launch_bounds__(256) k_pool_fwd(const PoolDesc* __restrict__ tab, const int* __restrict__ tstart,
                                                  int n) {
  const int inst = find_instance(tstart, n, blockIdx.x);
  const PoolDesc d = tab[inst];
  const int V = pool_vec(d.C);
  const int64_t i = ((int64_t)(blockIdx.x - tstart[inst]) * 256 + threadIdx.x) * V;
  if (i >= (int64_t)d.B * d.P * d.Q * d.C) return;
  if (V == 4) pool_fwd_at<4>(d, i);
  else pool_fwd_at<1>(d, i);
}

// dx[n,h,w,c] (+)= sum over windows whose first maximum sits at (h,w) of dy
template <int V>
__device__ __forceinline__ void pool_bwd_at(const PoolDesc& d, int64_t i) {
  const int c = (int)(i % d.C);
  int64_t t = i / d.C;
  const int w = (int)(t % d.W); t /= d.W;
  const int h = (int)(t % d.H);
  const int nb = (int)(t / d.H);
  const PoolSrc<V> src(d, c);
  float g[V];
#pragma unroll
  for (int j = 0; j < V; ++j) g[j] = 0.f;
  const int p_lo = max(0, (h + d.pad - d.k + d.stride) / d.stride), p_hi = min(d.P - 1, (h + d.pad) / d.stride);
  const int q_lo = max(0, (w + d.pad - d.k + d.stride) / d.stride), q_hi = min(d.Q - 1, (w + d.pad) / d.stride);
  for (int p = p_lo; p <= p_hi; ++p)
    for (int q = q_lo; q <= q_hi; ++q) {
      if (h + d.pad - p * d.stride >= d.k || w + d.pad - q * d.stride >= d.k) continue;
      float best[V];
      int at[V];  // position of the first maximum in the window
#pragma unroll
      for (int j = 0; j < V; ++j) { best[j] = -INFINITY; at[j] = -1; }
      for (int r = 0; r < d.k; ++r)
        for (int s = 0; s < d.k; ++s) {
          const int hh = p * d.stride + r - d.pad, ww = q * d.stride + s - d.pad;
          if (hh < 0 || hh >= d.H || ww < 0 || ww >= d.W) continue;
          float v[V];
          src.get((int64_t)(nb * d.H + hh) * d.W + ww, v);
#pragma unroll
          for (int j = 0; j < V; ++j)
            if (v[j] > best[j]) { best[j] = v[j]; at[j] = hh * d.W + ww; }
        }
      const float* dy = d.dy + ((int64_t)(nb * d.P + p) * d.Q + q) * d.C + c;
#pragma unroll
      for (int j = 0; j < V; ++j)
        if (at[j] == h * d.W + w) g[j] += __ldg(dy + j);
    }
#pragma unroll
  for (int j = 0; j < V; ++j) d.dx[i + j] = d.accumulate ? d.dx[i + j] + g[j] : g[j];
}
__global__ void __launch_bounds__(256) k_pool_bwd(const PoolDesc* __restrict__ tab, const int* __restrict__ tstart,
                                                  int n) {
  const int inst = find_instance(tstart, n, blockIdx.x);
  const PoolDesc d = tab[inst];
  const int V = pool_vec(d.C);
  const int64_t i = ((int64_t)(blockIdx.x - tstart[inst]) * 256 + threadIdx.x) * V;
  if (i >= (int64_t)d.B * d.H * d.W * d.C) return;
  if (V == 4) pool_bwd_at<4>(d, i);
  else pool_bwd_at<1>(d, i);
}

// ---------------------------------------------------------------- GEMM (head)
// C[m][n] = sum_k A[m][k] B[k][n] (+ bias[n]) (+ beta C[m][n]) (ReLU), fp32.
// BM x BN tiles by 128 threads of TM x TN outputs, 16-wide K steps, the next
// step's operands loaded into registers meanwhile, as float4 along whichever of
// an operand's two indices is contiguous (single elements at the edges and
// where the alignment does not allow it).  Bound by the fp32 FMA rate: with 8 x 8
// outputs a thread reads 64 bytes of shared memory for 64 FMAs -- with 4 x 4, as
// before, 32 for 16 -- and two FMAs are one packed instruction, which leaves the
// issue slots for the rest.  The K range of a tile is split over the CTAs of a
// cluster, so that a layer of 64 tiles still occupies every SM; the partial
// tiles meet in distributed shared memory and are added in rank order, each CTA
// finishing its share of the rows.  VGG-16's head at batch 128 (512 -> 4096 -> 4096
// -> 10): forward 0.50 -> 0.19 ms, backward 0.73 -> 0.37, with the head's small launches
// a third of the FMA rate (80 TFLOP/s).
template <int BM, int BN, int TM, int TN>
__global__ void __launch_bounds__(128, 4) k_gemm(const GemmDesc* __restrict__ desc) {
  constexpr int BK = 16, VM = TM < 4 ? TM : 4, VN = TN < 4 ? TN : 4;  // outputs in runs of VM rows, VN columns
  constexpr int TX = BN / TN;
  constexpr int UA = (BM * 4 + 127) / 128, UB = (BN * 4 + 127) / 128;  // float4 loads a thread and step
  static_assert(BM / TM * TX == 128, "128 threads");
  constexpr int PA = BM + 4, PB = BN + 4, PC = BN + 4;
  constexpr int kOperands = 2 * BK * (PA + PB), kTile = BM * PC;
  __shared__ __align__(16) float sm[kOperands > kTile ? kOperands : kTile];
  float* const As = sm;
  float* const Bs = sm + 2 * BK * PA;
  const GemmDesc d = *desc;
  uint32_t rank, splits;
  asm("mov.u32 %0, %cluster_ctarank;" : "=r"(rank));
  asm("mov.u32 %0, %cluster_nctarank;" : "=r"(splits));
  const int tile = blockIdx.x / splits, mt = (d.M + BM - 1) / BM;
  const int m0 = tile % mt * BM, n0 = tile / mt * BN;
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  const int kper = (d.K + (int)splits * BK - 1) / ((int)splits * BK) * BK;  // this CTA's share: whole steps
  const int kb0 = (int)rank * kper, kb1 = min(d.K, kb0 + kper);
  const bool a_k = d.sak == 1, b_k = d.sbk == 1;  // k contiguous in A / in B
  const bool a_v = ((a_k ? d.sam : d.sak) & 3) == 0 && (a_k || d.sam == 1) && (reinterpret_cast<uintptr_t>(d.A) & 15) == 0;
  const bool b_v = ((b_k ? d.sbn : d.sbk) & 3) == 0 && (b_k || d.sbn == 1) && (reinterpret_cast<uintptr_t>(d.Bm) & 15) == 0;
  float4 ra[UA], rb[UB];
  // four elements from (x, k) along k or along x
  auto load4 = [&](const float* p, int64_t sx, int64_t sk, int x, int X, int k, bool k_fast, bool vec) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (x >= X || k >= kb1) return v;
    p += x * sx + k * sk;
    if (vec && (k_fast ? k + 4 <= kb1 : x + 4 <= X)) return __ldg(reinterpret_cast<const float4*>(p));
    const int left = k_fast ? kb1 - k : X - x;
    const int64_t step = k_fast ? sk : sx;
    v.x = __ldg(p);
    if (left > 1) v.y = __ldg(p + step);
    if (left > 2) v.z = __ldg(p + 2 * step);
    if (left > 3) v.w = __ldg(p + 3 * step);
    return v;
  };
  auto load = [&](int k0) {
#pragma unroll
    for (int q = 0; q < UA; ++q) {
      const int u = tid + 128 * q;
      if (u < BM * 4)
        ra[q] = a_k ? load4(d.A, d.sam, d.sak, m0 + u / 4, d.M, k0 + u % 4 * 4, true, a_v)
                    : load4(d.A, d.sam, d.sak, m0 + u % (BM / 4) * 4, d.M, k0 + u / (BM / 4), false, a_v);
    }
#pragma unroll
    for (int q = 0; q < UB; ++q) {
      const int u = tid + 128 * q;
      if (u < BN * 4)
        rb[q] = b_k ? load4(d.Bm, d.sbn, d.sbk, n0 + u / 4, d.N, k0 + u % 4 * 4, true, b_v)
                    : load4(d.Bm, d.sbn, d.sbk, n0 + u % (BN / 4) * 4, d.N, k0 + u / (BN / 4), false, b_v);
    }
  };
  auto put = [&](float* s, int pitch, int W, int u, const float4& v, bool k_fast) {
    if (k_fast) {
      float* c = s + u % 4 * 4 * pitch + u / 4;
      c[0] = v.x; c[pitch] = v.y; c[2 * pitch] = v.z; c[3 * pitch] = v.w;
    } else {
      *reinterpret_cast<float4*>(s + u / (W / 4) * pitch + u % (W / 4) * 4) = v;
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int q = 0; q < UA; ++q)
      if (tid + 128 * q < BM * 4) put(As + buf * BK * PA, PA, BM, tid + 128 * q, ra[q], a_k);
#pragma unroll
    for (int q = 0; q < UB; ++q)
      if (tid + 128 * q < BN * 4) put(Bs + buf * BK * PB, PB, BN, tid + 128 * q, rb[q], b_k);
  };
  // output i of a thread is row BM / (TM / VM) * (i / VM) + VM ty + i % VM of the tile
  auto row = [&](int i) { return BM / (TM / VM) * (i / VM) + VM * ty + i % VM; };
  auto col = [&](int j) { return BN / (TN / VN) * (j / VN) + VN * tx + j % VN; };
  uint64_t acc[TM][TN / 2] = {};
  load(kb0);
  store(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = kb0; k0 < kb1; k0 += BK) {
    const bool more = k0 + BK < kb1;
    if (more) load(k0 + BK);
    const float* a0 = As + buf * BK * PA;
    const float* b0 = Bs + buf * BK * PB;
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      float av[TM];
      uint64_t bv[TN / 2];
#pragma unroll
      for (int i = 0; i < TM; i += VM) {
        if (VM == 4) *reinterpret_cast<float4*>(av + i) = *reinterpret_cast<const float4*>(a0 + kk * PA + row(i));
        else *reinterpret_cast<float2*>(av + i) = *reinterpret_cast<const float2*>(a0 + kk * PA + row(i));
      }
#pragma unroll
      for (int j = 0; j < TN; j += VN) {
        if (VN == 4) {
          const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(b0 + kk * PB + col(j));
          bv[j / 2] = v.x;
          bv[j / 2 + (VN == 4)] = v.y;
        } else {
          bv[j / 2] = *reinterpret_cast<const uint64_t*>(b0 + kk * PB + col(j));
        }
      }
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const uint64_t aa = tc::pk2(av[i], av[i]);
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) acc[i][j] = tc::fma2(aa, bv[j], acc[i][j]);
      }
    }
    if (more) store(buf ^ 1);
    __syncthreads();
    buf ^= 1;
  }
  // (a share past the end of K has read nothing and holds zeros)
  __syncthreads();
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; j += 2) *reinterpret_cast<uint64_t*>(sm + row(i) * PC + col(j)) = acc[i][j / 2];
  // every CTA of the cluster has left its sums; no one returns before this
  if (splits > 1) cluster_sync();
  else __syncthreads();
  const int rows = BM / (int)splits, r0 = (int)rank * rows;
  for (int e = tid; e < rows * BN; e += 128) {
    const int r = r0 + e / BN, c = e % BN;
    const int m = m0 + r, nc = n0 + c;
    if (m >= d.M || nc >= d.N) continue;
    float v = 0.f;
    for (uint32_t p = 0; p < splits; ++p) v += ld_cluster(sm + r * PC + c, p);
    if (d.bias) v += d.bias[nc];
    if (d.beta != 0.f) v += d.beta * d.Cm[(int64_t)m * d.scm + nc];
    if (d.relu) v = fmaxf(v, 0.f);
    d.Cm[(int64_t)m * d.scm + nc] = v;
  }
  if (splits > 1) {
    // a CTA's shared memory stays until its peers have read it
    __syncwarp();
    cluster_sync();
  }
}

// ---------------------------------------------------------------- head + misc
// One CTA per image and 32 channels: warp w adds pixels w, w + 8, ... (four in
// flight), the eight sums are added in warp order.  (A thread per channel over
// all pixels: 149 us for eight 32 x 32 x 16 images; the whole head
// forward now takes 38.)
__global__ void __launch_bounds__(256) k_gap(Src x, float* feat, int B, int HW, int C) {
  __shared__ float red[8][32];
  const int groups = (C + 31) / 32;
  const int b = blockIdx.x / groups, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = (blockIdx.x - b * groups) * 32 + lane;
  float s = 0.f;
  if (c < C) {
    int k = warp;
    for (; k + 24 < HW; k += 32) {
      float v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = ld_src(x, ((int64_t)b * HW + k + 8 * u) * C + c, c);
#pragma unroll
      for (int u = 0; u < 4; ++u) s += v[u];
    }
    for (; k < HW; k += 8) s += ld_src(x, ((int64_t)b * HW + k) * C + c, c);
  }
  red[warp][lane] = s;
  __syncthreads();
  if (warp == 0 && c < C) {
    float t = red[0][lane];
#pragma unroll
    for (int i = 1; i < 8; ++i) t += red[i][lane];
    feat[b * C + c] = t / (float)HW;
  }
}

// Sums over the rows of a group of HW, one after another (fp32 networks: average pool,
// bias gradients): out[b][c] = sum of x[b HW + k][c] / div.  32 columns a CTA; all
// warps bring 256 rows at a time to shared memory, the next ones in registers while one
// warp adds.  (One thread per sum with a load a row: 149 us for eight 32 x 32 x 16
// images.)
__global__ void __launch_bounds__(256) k_rowsum_fixed(Src x, float* out, int HW, int C, float div) {
  constexpr int R = 256, U = R / 8;
  __shared__ float tile[R][32];
  const int groups = (C + 31) / 32;
  const int b = blockIdx.x / groups, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = (blockIdx.x - b * groups) * 32 + lane;
  float v[U], s = 0.f;
  const float* p = static_cast<const float*>(x.ptr) + (int64_t)b * HW * C + c;  // (fp32 networks: DT_F32)
  const bool bn = c < C && x.scale != nullptr;
  const float sc = bn ? __ldg(x.scale + c) : 1.f, sf = bn ? __ldg(x.shift + c) : 0.f;
  auto load = [&](int k0) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int k = k0 + warp + 8 * u;
      v[u] = c < C && k < HW ? __ldg(p + (int64_t)k * C) : 0.f;
    }
  };
  load(0);
  for (int k0 = 0; k0 < HW; k0 += R) {
    __syncthreads();  // the previous rows have been added
#pragma unroll
    for (int u = 0; u < U; ++u) {
      float y = v[u];
      if (bn) {
        y = fmaf(sc, y, sf);
        if (x.relu) y = fmaxf(y, 0.f);
      }
      tile[warp + 8 * u][lane] = y;
    }
    __syncthreads();
    if (k0 + R < HW) load(k0 + R);
    if (warp == 0) {
      const int rows = min(R, HW - k0);
#pragma unroll 16
      for (int k = 0; k < rows; ++k) s += tile[k][lane];
    }
  }
  if (warp == 0 && c < C) out[(int64_t)b * C + c] = s / div;
}

__global__ void k_gap_bwd(const float* dfeat, float* dx, int B, int HW, int C) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)B * HW * C) return;
  const int c = (int)(i % C);
  const int b = (int)(i / ((int64_t)HW * C));
  dx[i] = dfeat[b * C + c] / (float)HW;
}

// one CTA: per-sample log-sum-exp loss (a warp per sample, up to 256 logits in
// registers), mean over the batch in a fixed order
constexpr int kCeThreads = 1024, kCeRegs = 8;
__global__ void __launch_bounds__(kCeThreads) k_softmax_ce(const float* logits, const int32_t* labels, int B, int m,
                                                           float* loss, float* dlogits, int32_t* status) {
  __shared__ float per[1024];
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const bool regs = m <= 32 * kCeRegs;
  for (int b = warp; b < B; b += kCeThreads / 32) {
    const float* z = logits + (int64_t)b * m;
    const int lab = labels[b];
    float zr[kCeRegs];
    float mx = -INFINITY;
    if (regs) {
#pragma unroll
      for (int i = 0; i < kCeRegs; ++i) zr[i] = lane + 32 * i < m ? z[lane + 32 * i] : -INFINITY;
#pragma unroll
      for (int i = 0; i < kCeRegs; ++i) mx = fmaxf(mx, zr[i]);
    } else {
      for (int i = lane; i < m; i += 32) mx = fmaxf(mx, z[i]);
    }
    for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    float se = 0.f;
    if (regs) {
#pragma unroll
      for (int i = 0; i < kCeRegs; ++i)
        if (lane + 32 * i < m) {
          se += expf(zr[i] - mx);
        }
    } else {
      for (int i = lane; i < m; i += 32) se += expf(z[i] - mx);
    }
    for (int off = 16; off > 0; off >>= 1) se += __shfl_xor_sync(0xffffffffu, se, off);
    const float lse = logf(se) + mx;
    if (regs) {
#pragma unroll
      for (int i = 0; i < kCeRegs; ++i) {
        const int j = lane + 32 * i;
        if (j < m) dlogits[(int64_t)b * m + j] = (expf(zr[i] - mx) / se - (j == lab ? 1.f : 0.f)) / (float)B;
      }
    } else {
      for (int i = lane; i < m; i += 32) {
        const float p = expf(z[i] - mx) / se;
        dlogits[(int64_t)b * m + i] = (p - (i == lab ? 1.f : 0.f)) / (float)B;
      }
    }
    if (lane == 0) per[b] = lse - ((lab >= 0 && lab < m) ? z[lab] : 0.f);
    if (lane == 0 && (lab < 0 || lab >= m)) atomicExch(status, 1);
  }
  __syncthreads();
  if (warp == 0) {
    double s = 0.0;
    for (int b = lane; b < B; b += 32) s += per[b];
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) {
      const float l = (float)(s / B);
      *loss = l;
      if (!isfinite(l)) atomicExch(status, 2);
    }
  }
}

// 32 columns a CTA; warp w adds rows w, w + 8, ..., the sums meet in warp order
__global__ void __launch_bounds__(256) k_colsum(const float* A, int rows, int cols, float* out) {
  __shared__ float red[8][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = blockIdx.x * 32 + lane;
  float s = 0.f;
  if (c < cols)
#pragma unroll 4
    for (int r = warp; r < rows; r += 8) s += __ldg(A + (int64_t)r * cols + c);
  red[warp][lane] = s;
  __syncthreads();
  if (warp == 0 && c < cols) {
    float t = red[0][lane];
#pragma unroll
    for (int i = 1; i < 8; ++i) t += red[i][lane];
    out[c] = t;
  }
}

__global__ void k_relu_mask(float* g, const float* pre, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n && !(pre[i] > 0.f)) g[i] = 0.f;
}

__global__ void k_sgd(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ v, void* shadow,
                      int32_t shadow_dt, int64_t n, float lr, float mu, float wd, int nesterov, int first) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const float wi = w[i];
    const float di = fmaf(wd, wi, g[i]);
    const float vi = first ? di : fmaf(mu, v[i], di);
    v[i] = vi;
    const float step = nesterov ? fmaf(mu, vi, di) : vi;
    const float wn = fmaf(-lr, step, wi);
    w[i] = wn;
    if (shadow) stv(shadow, shadow_dt, i, wn);
  }
}

__global__ void k_pack_input(const float* x, void* out, int32_t dt, int B, int C, int H, int W) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t total = (int64_t)B * C * H * W;
  if (i >= total) return;
  const int c = (int)(i % C);
  int64_t t = i / C;
  const int w = (int)(t % W); t /= W;
  const int h = (int)(t % H);
  const int b = (int)(t / H);
  stv(out, dt, i, x[(((int64_t)b * C + c) * H + h) * W + w]);
}

__global__ void k_export(Src x, int B, int H, int W, int C, float* out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t total = (int64_t)B * C * H * W;
  if (i >= total) return;
  const int c = (int)(i % C);
  int64_t t = i / C;
  const int w = (int)(t % W); t /= W;
  const int h = (int)(t % H);
  const int b = (int)(t / H);
  out[(((int64_t)b * C + c) * H + h) * W + w] = ld_src(x, i, c);
}

__global__ void k_copy_cast(const float* in, void* out, int32_t dt, int64_t n) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) stv(out, dt, i, in[i]);
}

// ---------------------------------------------------------------- launchers
static inline int cdiv64(int64_t a, int64_t b) { return (int)((a + b - 1) / b); }

namespace {
constexpr int kMaxDevices = 64;
std::atomic<int> g_sms[kMaxDevices];
std::atomic<uint32_t> g_attr_done[kMaxDevices];
std::mutex g_attr_mu;
}  // namespace

int device_sm_count() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 1;
  int v = g_sms[dev].load(std::memory_order_acquire);
  if (v > 0) return v;
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) return 1;
  g_sms[dev].store(sms, std::memory_order_release);
  return sms;
}

cudaError_t set_smem_attr_once(int slot, const void* kernel, int bytes) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices || slot < 0 || slot >= 32) return cudaErrorInvalidValue;
  const uint32_t bit = 1u << slot;
  if (g_attr_done[dev].load(std::memory_order_acquire) & bit) return cudaSuccess;
  std::lock_guard<std::mutex> lk(g_attr_mu);
  if (g_attr_done[dev].load(std::memory_order_acquire) & bit) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) g_attr_done[dev].fetch_or(bit, std::memory_order_release);
  return e;
}

cudaError_t launch_conv_fwd_simt(const ConvDesc* tab, const int* tstart, int n, int total, int variant,
                                 cudaStream_t st) {
  if (total <= 0) return cudaSuccess;
  if (variant == 0) k_conv_fwd<64, 64><<<total, 256, 0, st>>>(tab, tstart, n);
  else if (variant == 1) k_conv_fwd<128, 32><<<total, 256, 0, st>>>(tab, tstart, n);
  else if (variant == 2) k_conv_fwd<64, 16><<<total, 256, 0, st>>>(tab, tstart, n);
  else if (variant == 4) k_conv_fwd_quad<<<total, 256, 0, st>>>(tab, tstart, n);
  else k_conv_fwd_few<<<total, 256, 0, st>>>(tab, tstart, n);
  return cudaGetLastError();
}
cudaError_t launch_conv_dgrad_simt(const ConvDesc* tab, const int* tstart, int n, int total, int variant,
                                   cudaStream_t st) {
  if (total <= 0) return cudaSuccess;
  if (variant == 0) k_conv_dgrad<64, 64><<<total, 256, 0, st>>>(tab, tstart, n);
  else if (variant == 1) k_conv_dgrad<128, 32><<<total, 256, 0, st>>>(tab, tstart, n);
  else k_conv_dgrad<64, 16><<<total, 256, 0, st>>>(tab, tstart, n);
  return cudaGetLastError();
}
cudaError_t launch_conv_wgrad_simt(const ConvDesc* tab, const int* tstart, int n, int total, int variant,
                                   cudaStream_t st) {
  if (total <= 0) return cudaSuccess;
  if (variant == 0) k_conv_wgrad<64><<<total, 256, 0, st>>>(tab, tstart, n);
  else if (variant == 1) k_conv_wgrad<16><<<total, 256, 0, st>>>(tab, tstart, n);
  else if (variant == 2) k_conv_wgrad_few<16><<<total, 256, 0, st>>>(tab, tstart, n);
  else if (variant == 3) k_conv_wgrad_few<32><<<total, 256, 0, st>>>(tab, tstart, n);
  else k_conv_wgrad_few1<<<total, 256, 0, st>>>(tab, tstart, n);
  return cudaGetLastError();
}
cudaError_t launch_wreduce(const WReduceDesc* tab, const int* tstart, int n, int total, cudaStream_t st) {
  if (total <= 0) return cudaSuccess;
  k_wreduce<<<total, 256, 0, st>>>(tab, tstart, n);
  return cudaGetLastError();
}
cudaError_t launch_wtrans(const WtDesc* tab, const int* tstart, int n, int total, cudaStream_t st) {
  if (total <= 0) return cudaSuccess;
  k_wtrans<<<total, 256, 0, st>>>(tab, tstart, n);
  return cudaGetLastError();
}
cudaError_t launch_ew(const EwDesc* tab, const int* tstart, int n, int total, cudaStream_t st) {
  if (total <= 0) return cudaSuccess;
  k_ew<<<total, 256, 0, st>>>(tab, tstart, n);
  return cudaGetLastError();
}
cudaError_t launch_ew_bwd(const EwBwdDesc* tab, const int* tstart, int n, int total, cudaStream_t st) {
  if (total <= 0) return cudaSuccess;
  k_ew_bwd<<<total, 256, 0, st>>>(tab, tstart, n);
  return cudaGetLastError();
}
cudaError_t launch_bn_fin(const BnFinDesc* tab, const int* tstart, int n, int total, int fixed_order, cudaStream_t st) {
  if (total <= 0) return cudaSuccess;
  if (fixed_order) k_bn_fin<true><<<total, kFinThreads, 0, st>>>(tab, tstart, n);
  else k_bn_fin<false><<<total, kFinThreads, 0, st>>>(tab, tstart, n);
  return cudaGetLastError();
}
cudaError_t launch_bn_eval(const BnFinDesc* tab, const int* tstart, int n, int total, cudaStream_t st) {
  if (total <= 0) return cudaSuccess;
  k_bn_eval<<<total, kFinEvalChannels, 0, st>>>(tab, tstart, n);
  return cudaGetLastError();
}
cudaError_t launch_bnb_reduce(const BnBwdDesc* tab, const int* tstart, int n, int total, cudaStream_t st) {
  if (total <= 0) return cudaSuccess;
  k_bnb_reduce<<<total, 256, 0, st>>>(tab, tstart, n);
  return cudaGetLastError();
}
cudaError_t launch_bnb_reduce8(const BnBwdDesc* tab, const int* tstart, int n, int total, cudaStream_t st) {
  if (total <= 0) return cudaSuccess;
  k_bnb_reduce8<<<total, 256, 0, st>>>(tab, tstart, n);
  return cudaGetLastError();
}
cudaError_t launch_bnb_reduce_fixed(const BnBwdDesc* tab, const int* tstart, int n, int total, cudaStream_t st) {
  if (total <= 0) return cudaSuccess;
  k_bnb_reduce_fixed<<<total, 256, 0, st>>>(tab, tstart, n);
  return cudaGetLastError();
}
cudaError_t launch_bnb_fin(const BnBwdDesc* tab, const int* tstart, int n, int total, cudaStream_t st) {
  if (total <= 0) return cudaSuccess;
  k_bnb_fin<<<total, kFinThreads, 0, st>>>(tab, tstart, n);
  return cudaGetLastError();
}
cudaError_t launch_bnb_apply(const BnBwdDesc* tab, const int* tstart, int n, int total, cudaStream_t st) {
  if (total <= 0) return cudaSuccess;
  k_bnb_apply<<<total, 256, 0, st>>>(tab, tstart, n);
  return cudaGetLastError();
}
cudaError_t launch_bnb_apply8(const BnBwdDesc* tab, const int* tstart, int n, int total, cudaStream_t st) {
  if (total <= 0) return cudaSuccess;
  k_bnb_apply8<<<total, 256, 0, st>>>(tab, tstart, n);
  return cudaGetLastError();
}
cudaError_t launch_pool_fwd(const PoolDesc* tab, const int* tstart, int n, int total, cudaStream_t st) {
  if (total <= 0) return cudaSuccess;
  k_pool_fwd<<<total, 256, 0, st>>>(tab, tstart, n);
  return cudaGetLastError();
}
cudaError_t launch_pool_bwd(const PoolDesc* tab, const int* tstart, int n, int total, cudaStream_t st) {
  if (total <= 0) return cudaSuccess;
  k_pool_bwd<<<total, 256, 0, st>>>(tab, tstart, n);
  return cudaGetLastError();
}
cudaError_t launch_gemm(const GemmDesc* desc, int M, int N, int K, int fixed_order, cudaStream_t st) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  // 32 x 16 tiles where a 128 x 64 tile would be mostly padding (a classifier's
  // few columns)
  const bool small = M <= 32 || N <= 16;
  int BM = small ? 32 : 128, BN = small ? 16 : 64;
  auto count = [&]() { return (int64_t)((M + BM - 1) / BM) * ((N + BN - 1) / BN); };
  // a sum of an fp32 network is not split: smaller tiles where the large ones leave SMs idle
  const bool mid = fixed_order && !small && count() < device_sm_count();
  if (mid) BM = 64, BN = 32;
  const int64_t tiles = count();
  // CTAs of a tile: while the launch fits the chip at once (four CTAs an SM) and
  // each keeps at least 128 of K
  int splits = 1;
  while (!fixed_order && splits < 8 && tiles * splits * 2 <= 4 * (int64_t)device_sm_count() && K / (splits * 2) >= 128) splits *= 2;
  if (tiles * splits > 0x7fffffff) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(tiles * splits));
  cfg.blockDim = dim3(128);
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = splits;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  const cudaError_t e = small ? cudaLaunchKernelEx(&cfg, k_gemm<32, 16, 2, 2>, desc)
                        : mid ? cudaLaunchKernelEx(&cfg, k_gemm<64, 32, 4, 4>, desc)
                              : cudaLaunchKernelEx(&cfg, k_gemm<128, 64, 8, 8>, desc);
  return e != cudaSuccess ? e : cudaGetLastError();
}
cudaError_t launch_pack_input(const float* x, void* out, int32_t dt, int B, int C, int H, int W, cudaStream_t st) {
  const int64_t total = (int64_t)B * C * H * W;
  k_pack_input<<<cdiv64(total, 256), 256, 0, st>>>(x, out, dt, B, C, H, W);
  return cudaGetLastError();
}
cudaError_t launch_gap(Src x, float* feat, int B, int HW, int C, int fixed_order, cudaStream_t st) {
  if (fixed_order) k_rowsum_fixed<<<B * cdiv64(C, 32), 256, 0, st>>>(x, feat, HW, C, (float)HW);
  else k_gap<<<B * cdiv64(C, 32), 256, 0, st>>>(x, feat, B, HW, C);
  return cudaGetLastError();
}
cudaError_t launch_gap_bwd(const float* dfeat, float* dx, int B, int HW, int C, cudaStream_t st) {
  k_gap_bwd<<<cdiv64((int64_t)B * HW * C, 256), 256, 0, st>>>(dfeat, dx, B, HW, C);
  return cudaGetLastError();
}
cudaError_t launch_softmax_ce(const float* logits, const int32_t* labels, int B, int m, float* loss,
                              float* dlogits, int32_t* status, cudaStream_t st) {
  if (B > 1024) return cudaErrorInvalidValue;
  k_softmax_ce<<<1, kCeThreads, 0, st>>>(logits, labels, B, m, loss, dlogits, status);
  return cudaGetLastError();
}
cudaError_t launch_colsum(const float* A, int rows, int cols, float* out, int fixed_order, cudaStream_t st) {
  if (fixed_order) k_rowsum_fixed<<<cdiv64(cols, 32), 256, 0, st>>>(Src{A, nullptr, nullptr, DT_F32, 0}, out, rows, cols, 1.f);
  else k_colsum<<<cdiv64(cols, 32), 256, 0, st>>>(A, rows, cols, out);
  return cudaGetLastError();
}
cudaError_t launch_relu_mask(float* g, const float* pre, int64_t n, cudaStream_t st) {
  k_relu_mask<<<cdiv64(n, 256), 256, 0, st>>>(g, pre, n);
  return cudaGetLastError();
}
cudaError_t launch_sgd(float* w, const float* g, float* v, void* shadow, int32_t shadow_dt, int64_t n, float lr,
                       float mu, float wd, int nesterov, int first, cudaStream_t st) {
  int blocks = cdiv64(n, 256);
  if (blocks > device_sm_count() * 16) blocks = device_sm_count() * 16;
  if (blocks < 1) blocks = 1;
  k_sgd<<<blocks, 256, 0, st>>>(w, g, v, shadow, shadow_dt, n, lr, mu, wd, nesterov, first);
  return cudaGetLastError();
}
cudaError_t launch_export(Src x, int B, int H, int W, int C, float* out, cudaStream_t st) {
  const int64_t total = (int64_t)B * C * H * W;
  k_export<<<cdiv64(total, 256), 256, 0, st>>>(x, B, H, W, C, out);
  return cudaGetLastError();
}
cudaError_t launch_copy_cast(const float* in, void* out, int32_t dt, int64_t n, cudaStream_t st) {
  int blocks = cdiv64(n, 256);
  if (blocks > device_sm_count() * 16) blocks = device_sm_count() * 16;
  if (blocks < 1) blocks = 1;
  k_copy_cast<<<blocks, 256, 0, st>>>(in, out, dt, n);
  return cudaGetLastError();
}
cudaError_t launch_weight_cast(const float* in, void* out, int32_t dt, int64_t n, cudaStream_t st) {
  return launch_copy_cast(in, out, dt, n, st);
}

}  // namespace pnn
