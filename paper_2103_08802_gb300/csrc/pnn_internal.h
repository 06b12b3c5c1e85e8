// Internal descriptors shared by the host runtime and the CUDA kernels.
// Every grouped launch receives a device table of per-instance descriptors
// plus a prefix array of tile counts; CTA b belongs to the instance i with
// tile_start[i] <= b < tile_start[i+1].  Tensors are NHWC with the batch
// folded into the row index (row m = (n*H + h)*W + w).
#pragma once
#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#ifdef __CUDACC__
#define PNN_HD __host__ __device__
#else
#define PNN_HD
#endif

namespace pnn {

enum DType : int32_t { DT_F32 = 0, DT_BF16 = 1 };

// A tensor operand.  When scale != nullptr the value read is the "virtual"
// BN(+ReLU) output  v = act(scale[c] * src + shift[c]); zero padding of a
// convolution applies to v, not to src.
struct Src {
  const void* ptr;
  const float* scale;
  const float* shift;
  int32_t dt;
  int32_t relu;
};

struct ConvDesc {
  Src x;                 // forward / wgrad: conv input (maybe virtual)
  const void* w;         // weights [K][R][S][C], dtype w_dt
  int32_t w_dt;
  int32_t B, H, W, C;    // input geometry
  int32_t P, Q, K;       // output geometry
  int32_t R, S, stride, pad;
  // forward epilogue
  void* y; int32_t y_dt;
  const void* res; int32_t res_dt;   // residual added to the output (or null)
  // up to two more addends, out += res2_c[e] * res2[e] (null: none): the
  // parareal correction folded into the conv that produces its operand
  // (r_j = y_j - x_{j+1}, rt_{j+1} = r_{j+1} + F^j(rt_j), ytilde = y_N + rt_N)
  const void* res2[2]; int32_t res2_dt[2]; float res2_c[2];
  float* stats;                       // per-tile BN partials [mtiles][K][2] = (mean, M2) or null
  int32_t stat_rows;                  // k_conv_fwd_few: rows of a partial (fp32 networks), or 0: the CTA's
  // dgrad: dx[B*H*W][C] (fp32) = (accumulate ? dx : 0) + W^T * dy
  float* dx; int32_t accumulate;
  // dgrad / wgrad operand dy[B*P*Q][K] (fp32)
  const float* dy;
  // wgrad: partial sums [splits][K][R*S*C]
  float* dw_part;
  int32_t splits, pix_per_split;
  int32_t mtiles, ntiles;             // tile grid of this instance
  int32_t ntile_w;                    // N columns of a tile when ntiles > 1 (256, or 128 TMA-fed)
  int32_t mtile_rows;                 // M rows of a tile: 128, or 256 (TMA-fed weight gradient: two MMA halves)
  int32_t op_bf16;                    // round both contraction operands to bf16 (bf16 mode)
  // TMA-fed tensor-core variant (stride 1): device addresses of two 2-D tensor
  // maps (CUtensorMap, 128-byte aligned) -- tma_a over the A source rows
  // [pixels][channels] (forward: x, dgrad: dy; box min(channels, 64) x 128,
  // no swizzle), tma_b over the bf16 weight rows [N][K] (box 64 x BN,
  // 128-byte swizzle)
  const void* tma_a;
  const void* tma_b;
  // TMA-fed 3x3 forward / data gradient whose tiles lie inside one image
  // (halo_ok): tensor map over the same A source rows with box [halo_rows(W)
  // rows x channels] (no swizzle) -- one box per tile covers all nine taps
  // (null: one box per tap)
  const void* tma_h;
  // TMA-fed forward: tensor map over the output y [pixels][K] (box 16
  // columns x 32 rows, 64-byte swizzle for fp32, 32-byte for bf16), or null
  const void* tma_y;
  // k_pw_conv.cu, k_c3_conv.cu: tensor map over the unit's second operand
  // (forward: the residual, data gradient: the BN input h) with box [128 rows x
  // unit columns] bf16; ntile_w is then (1x1) the columns of an item
  const void* tma_x;
  // TMA-fed data gradient of a BN(+ReLU) value (x = that virtual value): when
  // bnb_part is set, the epilogue also writes the BN-backward partial sums of
  // its tile, [m-tile][C][2] = (sum g, sum g * xhat) with g = dA masked by the
  // ReLU and xhat = (h - mean) * rstd
  const float* bn_mean;
  const float* bn_rstd;
  float* bnb_part;
};

// out = act( sum_i coef_i * in_i ), optional BN partials of out, NHWC [M][C].
struct EwDesc {
  Src in[3];
  float coef[3];
  int32_t nin;
  void* out; int32_t out_dt;
  int32_t relu;
  float* stats;          // [tiles][C][2] = (mean, M2) or null
  int64_t M;
  int32_t C;
  int32_t rows_per_tile;
  int32_t groups;        // row groups of a channel's partials, or 0: as many as the CTA's threads give
};

// backward of EW: g = dout * [out > 0 if relu]; grad_i (+)= coef_i * g
struct EwBwdDesc {
  const float* dout;
  const void* out; int32_t out_dt; int32_t relu;
  float* gin[3]; float coef[3]; int32_t acc[3];
  int32_t nin;
  int64_t M; int32_t C;
};

// BN statistics finalisation: partials[tiles][C][2] -> mean, rstd, scale, shift
constexpr int kFinChannels = 8;       // BN finalize: channels a CTA
constexpr int kFinEvalChannels = 256; // eval mode: channels a CTA
inline int fin_ctas(int C) { return (C + kFinChannels - 1) / kFinChannels; }
struct BnFinDesc {
  const float* part;     // [tiles][C][2] = (mean, M2) of each tile's rows
  int32_t tiles, C;
  int64_t count;         // number of rows M
  int32_t rows_per_tile; // rows of every partial tile but the last
  const float* gamma; const float* beta;
  float* mean; float* rstd; float* scale; float* shift;
  float* run_mean; float* run_var;  // running statistics of this BN layer
  float momentum;                   // training: rate at which they follow the batch
  double inv_count;                 // 1 / count
};

// BN backward: dz = da * [z > 0 if relu], z = scale*h + shift, xhat = (h-mean)*rstd
//   reduce: part[tile][c] = (sum dz, sum dz*xhat)
//   fin:    dbeta = sum dz, dgamma = sum dz*xhat, coef[c] = (gamma*rstd, dbeta/M, dgamma/M)
//   apply:  dh (+)= gamma*rstd * (dz - dbeta/M - xhat*dgamma/M)
struct BnBwdDesc {
  const float* da;
  const void* h; int32_t h_dt;
  const float* mean; const float* rstd; const float* scale; const float* shift;
  const float* gamma;
  int32_t relu;
  float* part;           // [tiles][C][2]
  float* dgamma; float* dbeta;
  float* coef;           // [C][3]
  float* dh; int32_t accumulate;     // apply: accumulate into dh; fin: into dgamma/dbeta
  const float* add0; const float* add1;  // apply: extra gradients added into dh (residual paths)
  float add_c[2];                          // their coefficients
  int64_t M; int32_t C;
  int32_t rows_per_tile, tiles;
  double inv_count;                        // fin: 1 / M
};

PNN_HD inline int pool_vec(int C) { return C % 4 == 0 ? 4 : 1; }  // channels a thread
struct PoolDesc {
  Src x;                 // input (maybe virtual)
  void* y; int32_t y_dt; // output
  int32_t B, H, W, C, P, Q, k, stride, pad;
  // backward: dx (+)= route(dy)
  const float* dy; float* dx; int32_t accumulate;
  int32_t tiles;
};

// wgrad split reduction: dw[K*RSC] = sum_s part[s][...]; partials are laid out
// [s][K][RSC] or [s][RSC][K] (transposed = 1)
constexpr int kWreduceElems = 128;  // elements a CTA
struct WReduceDesc {
  const float* part;
  float* dw;
  int32_t splits;
  int32_t accumulate;
  int64_t n;
  int32_t tiles;
  int32_t transposed, kout, rsc;
};

// bf16 weight copies from src[K][RS][C].  pack 0: dst[c][r][s][k], for the
// tensor-core data gradient.  pack 1 (forward: rows n = k, channels ch = c) and 2
// (data gradient: n = c, ch = k): the operand layout of k_c3_conv.cu,
// dst[n / 64][ch / 8][tap][n % 64][ch % 8]
struct WtDesc {
  const void* src;
  void* dst;
  int32_t K, RS, C, pack;
  int64_t n;
};
// CTAs of k_wtrans for it: an element a thread, or (packed) eight
inline int wtrans_ctas(const WtDesc& w) { return (int)(((w.pack ? w.n / 8 : w.n) + 255) / 256); }

// generic strided fp32 GEMM: C[m][n] = beta*C + sum_k A[m*sam + k*sak] * B[k*sbk + n*sbn] (+ bias[n]) (relu)
struct GemmDesc {
  const float* A; const float* Bm; float* Cm;
  const float* bias;
  int32_t M, N, K;
  int64_t sam, sak, sbk, sbn, scm;
  float beta;
  int32_t relu;
};

// ------------------------------------------------------------ launchers
// All launchers enqueue on `st` and return cudaGetLastError().
cudaError_t launch_conv_fwd_simt(const ConvDesc* tab, const int* tstart, int n, int total_tiles,
                                 int variant, cudaStream_t st);
cudaError_t launch_conv_dgrad_simt(const ConvDesc* tab, const int* tstart, int n, int total_tiles,
                                   int variant, cudaStream_t st);
// variant: simt_wgrad_variant
cudaError_t launch_conv_wgrad_simt(const ConvDesc* tab, const int* tstart, int n, int total_tiles, int variant,
                                   cudaStream_t st);
cudaError_t launch_wreduce(const WReduceDesc* tab, const int* tstart, int n, int total_tiles, cudaStream_t st);
cudaError_t launch_ew(const EwDesc* tab, const int* tstart, int n, int total_tiles, cudaStream_t st);
cudaError_t launch_ew_bwd(const EwBwdDesc* tab, const int* tstart, int n, int total_tiles, cudaStream_t st);
cudaError_t launch_bn_fin(const BnFinDesc* tab, const int* tstart, int n, int total_tiles, int fixed_order,
                          cudaStream_t st);
// eval mode: scale and shift from the running statistics (total: CTAs of kFinEvalChannels channels)
cudaError_t launch_bn_eval(const BnFinDesc* tab, const int* tstart, int n, int total, cudaStream_t st);
cudaError_t launch_bnb_reduce(const BnBwdDesc* tab, const int* tstart, int n, int total_tiles, cudaStream_t st);
cudaError_t launch_bnb_fin(const BnBwdDesc* tab, const int* tstart, int n, int total_tiles, cudaStream_t st);
cudaError_t launch_bnb_apply(const BnBwdDesc* tab, const int* tstart, int n, int total_tiles, cudaStream_t st);
// 8 channels per thread; every instance needs C % 8 == 0 and C <= 2048
cudaError_t launch_bnb_reduce8(const BnBwdDesc* tab, const int* tstart, int n, int total_tiles, cudaStream_t st);
// fp32 networks; total: two CTAs a tile
cudaError_t launch_bnb_reduce_fixed(const BnBwdDesc* tab, const int* tstart, int n, int total, cudaStream_t st);
cudaError_t launch_bnb_apply8(const BnBwdDesc* tab, const int* tstart, int n, int total_tiles, cudaStream_t st);
cudaError_t launch_pool_fwd(const PoolDesc* tab, const int* tstart, int n, int total_tiles, cudaStream_t st);
cudaError_t launch_pool_bwd(const PoolDesc* tab, const int* tstart, int n, int total_tiles, cudaStream_t st);
// desc (device memory) of an M x N x K product
cudaError_t launch_gemm(const GemmDesc* desc, int M, int N, int K, int fixed_order, cudaStream_t st);
// tcgen05 implicit-GEMM convolution (bf16 operands, fp32 accumulate in TMEM);
// instances need C % 8 == 0; bnmax = largest N tile (multiple of 16, <= 256)
// (max_ctas > 0 caps the persistent grid below the SM count, leaving SMs to
// launches of other streams)
cudaError_t launch_conv_fwd_tc(const ConvDesc* tab, const int* tstart, int n, int total_tiles, int bnmax,
                               int32_t* status, cudaStream_t st, int max_ctas = 0);
cudaError_t launch_conv_dgrad_tc(const ConvDesc* tab, const int* tstart, int n, int total_tiles, int bnmax,
                                 int32_t* status, cudaStream_t st, int max_ctas = 0);
cudaError_t launch_conv_wgrad_tc(const ConvDesc* tab, const int* tstart, int n, int total_tiles, int bnmax,
                                 int32_t* status, cudaStream_t st, int max_ctas = 0);
// TMA-fed stride-1 forward (mode 0), data-gradient (mode 1) or weight-gradient
// (mode 2) tensor-core conv; raw_bytes: one pipeline stage's raw slot (the
// largest over the launch's instances, a multiple of 1024); op_bytes: one
// stage's operand slot when the launch has halo tiles (the larger of
// halo_op_bytes and the default slot), 0 for the default slot
// wide: every tile of the launch is one k-step (the epilogue bounds the
// kernel): the variant with three epilogue groups and two transform warps
cudaError_t launch_conv_tma(int mode, int wide, const ConvDesc* tab, const int* tstart, int n, int total, int bnmax,
                            int raw_bytes, int op_bytes, int32_t* status, cudaStream_t st, int max_ctas = 0);
// whether the TMA-fed kernel of `mode` holds at least two stages of this size
bool conv_tma_fits(int mode, int bnmax, int raw_bytes, int op_bytes = 0);
// the default operand slot of a TMA-fed stage (A then bnmax weight rows)
int conv_tma_op_bytes(int mode, int bnmax);
// whether a halo instance (mode 0 or 1; A source W x ch, N tile bn) leaves
// two stages even beside per-tap instances of the same launch
bool conv_halo_fits(int mode, int W, int ch, int bn);
// 1x1 stride-1 forward (mode 0) / data gradient (mode 1) of k_pw_conv.cu;
// total: items; raw_bytes, x_bytes: the largest raw A slot and second operand
// over the launch's instances (multiples of 1024); wide: every instance has one
// k-step and at least 64 output columns
cudaError_t launch_conv_pw(int mode, int wide, const ConvDesc* tab, const int* ts, int total, int raw_bytes,
                           int x_bytes, int32_t* status, cudaStream_t st, int max_ctas = 0);
// 3x3 stride-1 forward (mode 0) / data gradient (mode 1) of k_c3_conv.cu; s: the
// largest slots over the launch's instances (c3_add)
struct C3Slots;
cudaError_t launch_conv_c3(int mode, const ConvDesc* tab, const int* ts, int total, const C3Slots& s,
                           int32_t* status, cudaStream_t st, int max_ctas = 0);
// weight gradient of k_wg_conv.cu; any: wg_any of some instance; raw_bytes, op_bytes:
// the largest slots over the launch's instances (multiples of 1024)
cudaError_t launch_conv_wg(int ksize, int any, const ConvDesc* tab, const int* ts, int total, int raw_bytes, int op_bytes,
                           int32_t* status, cudaStream_t st, int max_ctas = 0);
// record a message for pnn_last_error(NULL) and return `code`
int set_last_error(int code, const char* msg);
// streaming multiprocessors of the current device, queried once per device
// (thread-safe); 1 if the query fails, which keeps every grid valid
int device_sm_count();
// cudaFuncSetAttribute(MaxDynamicSharedMemorySize) once per (device, kernel
// slot < 32); thread-safe
cudaError_t set_smem_attr_once(int slot, const void* kernel, int bytes);

// debug builds: first misaligned vector access of the tensor-core kernels (0 = none)
unsigned long long conv_tc_debug_word();
cudaError_t launch_wtrans(const WtDesc* tab, const int* tstart, int n, int total_tiles, cudaStream_t st);
constexpr int kTcBM = 128;

// single-instance helpers
cudaError_t launch_pack_input(const float* x_nchw, void* out, int32_t out_dt, int B, int C, int H, int W,
                              cudaStream_t st);
cudaError_t launch_gap(Src x, float* feat, int B, int HW, int C, int fixed_order, cudaStream_t st);
cudaError_t launch_gap_bwd(const float* dfeat, float* dx, int B, int HW, int C, cudaStream_t st);
cudaError_t launch_softmax_ce(const float* logits, const int32_t* labels, int B, int m, float* loss,
                              float* dlogits, int32_t* status, cudaStream_t st);
cudaError_t launch_colsum(const float* A, int rows, int cols, float* out, int fixed_order, cudaStream_t st);
cudaError_t launch_relu_mask(float* g, const float* pre, int64_t n, cudaStream_t st);
cudaError_t launch_sgd(float* w, const float* g, float* v, void* shadow, int32_t shadow_dt, int64_t n,
                       float lr, float mu, float wd, int nesterov, int first, cudaStream_t st);
cudaError_t launch_export(Src x, int B, int H, int W, int C, float* out_nchw, cudaStream_t st);
cudaError_t launch_copy_cast(const float* in, void* out, int32_t out_dt, int64_t n, cudaStream_t st);
cudaError_t launch_weight_cast(const float* in, void* out, int32_t out_dt, int64_t n, cudaStream_t st);

// tile geometry helpers shared by runtime and kernels
constexpr int kEwRowsPerTile = 64;
// channels of a CTA of the elementwise sum, and its CTAs a row tile
constexpr int kEwSlice = 64;
PNN_HD inline int ew_slices(int C) { return (C + kEwSlice - 1) / kEwSlice; }
// row groups of its BN partials in an fp32 network (see "Fixed order", k_simt.cu)
inline int ew_fixed_groups(int C) { return C <= 256 ? 256 / C : 1; }
// elements of a CTA of its gradient: 64 rows, of a wide layer fewer (with 64 rows of
// 512 channels the six launches of a VGG-16 step took 124 us, now 56)
PNN_HD inline int ew_bwd_elems(int C) { return C < 64 ? kEwRowsPerTile * C : 4096; }
// BN forward statistics are kept as (count, mean, M2 = sum of squared
// deviations from the mean) and combined with the pairwise update of Chan,
// Golub & LeVeque ("Updating formulae and a pairwise algorithm for computing
// sample variances", 1979): for disjoint sets a and b with n = n_a + n_b and
// delta = mean_b - mean_a,
//   mean = mean_a + delta * n_b / n,   M2 = M2_a + M2_b + delta^2 * n_a * n_b / n,
// which never subtracts two large sums (the one-pass sum(h^2) - n * mean^2
// loses the variance when |mean| >> std).  Per-tile partials are
// [tiles][C][2] = (mean, M2) of the tile's rows; a tile's count follows from
// its row range.
template <typename T>
PNN_HD inline void chan_merge(T& n, T& mean, T& m2, T nb, T meanb, T m2b) {
  if (nb <= T(0)) return;
  if (n <= T(0)) { n = nb; mean = meanb; m2 = m2b; return; }
  const T nn = n + nb;
  const T delta = meanb - mean;
  const T f = nb / nn;
  mean = mean + delta * f;
  m2 = m2 + m2b + delta * delta * n * f;
  n = nn;
}

// TMA-fed weight gradient: the two boxes of a k-step (64 pixels) -- the
// activation rows of every tap (halo of pad*W + pad rows each side) x cwx
// channels, and the output-gradient rows x K -- and their raw-slot offsets
struct WgBoxes {
  int halo, hrows, cwx, escx, xbytes, yoff, ybytes;
};
PNN_HD inline WgBoxes wg_boxes(int C, int K, int W, int pad, bool xbf) {
  WgBoxes b;
  b.halo = pad * W + pad;
  b.hrows = 64 + 2 * b.halo;
  b.cwx = C <= 64 ? C : 128;
  b.escx = xbf ? 2 : 4;
  b.xbytes = b.hrows * b.cwx * b.escx;
  b.yoff = (b.xbytes + 127) & ~127;
  b.ybytes = 64 * K * 4;
  return b;
}
PNN_HD inline int wg_raw_bytes(const WgBoxes& b) { return (b.yoff + b.ybytes + 1023) & ~1023; }

// TMA-fed 3x3 forward / data gradient, halo tiles.  A 128-pixel tile that
// lies inside one image reads input pixels m0 - W - 1 .. m0 + 128 + W: one
// box of halo_rows(W) rows.  The transform forms three copies of it, one per
// column offset s' in {-1, 0, 1}, each of 128 + 2W rows (copy s' row j =
// pixel m0 - W + s' + j, zero where that pixel lies outside the tile's image
// or where the output column x - s' would leave the row), in the
// no-swizzle K-major layout: one plane of 16-byte rows per 8 channels.  Tap
// (r', s') is then copy s' from row (r' + 1) W: a descriptor offset, for any
// W.  Needs 128 | H*W (no tile crosses an image), W <= 63 (a TMA box holds
// at most 256 rows) and 16 | channels <= 64.
PNN_HD inline bool halo_ok(int k, int stride, int pad, int H, int W, int ch) {
  return k == 3 && stride == 1 && pad == 1 && W > 0 && (H * W) % kTcBM == 0 && kTcBM + 2 * W + 2 <= 256 &&
         ch % 16 == 0 && ch <= 64;
}
PNN_HD inline int halo_rows(int W) { return kTcBM + 2 * W + 2; }
PNN_HD inline int halo_plane_bytes(int W) { return (kTcBM + 2 * W) * 16; }
PNN_HD inline int halo_copy_bytes(int W, int ch) { return (ch / 8) * halo_plane_bytes(W); }
// weight boxes of a halo tile: the tile's whole K = 9 * ch in boxes of 64
PNN_HD inline int halo_nbox(int ch) { return (9 * ch + 63) / 64; }
PNN_HD inline int halo_raw_bytes(int W, int ch, int esz) { return (halo_rows(W) * ch * esz + 1023) & ~1023; }
// operand slot of a halo tile: the weight boxes (bn rows each), then the three copies
PNN_HD inline int halo_op_bytes(int W, int ch, int bn) {
  return (halo_nbox(ch) * bn * 128 + 3 * halo_copy_bytes(W, ch) + 1023) & ~1023;
}

// ---------------------------------------------------------------- conv kernel choice
// (mode 0 forward, 1 data gradient, 2 weight gradient; variant 1 = TMA-fed,
// 0 = thread-gathered tensor-core kernel)
// The TMA-fed forward / data gradient load each filter tap as one
// [128 rows x min(channels, 64)] box: stride 1, same padding, and a channel
// count (of the A source) that divides 64 or is a multiple of it.
inline bool tma_shape_ok(int k, int stride, int pad, int ch) {
  const bool geom = stride == 1 && ((k == 1 && pad == 0) || (k == 3 && pad == 1));
  return geom && ch % 8 == 0 && (ch <= 64 ? 64 % ch == 0 : ch % 64 == 0);
}
// 1x1 stride-1 forward / data gradient of k_pw_conv.cu (variant 4): ch
// channels of the A source, ncols GEMM columns.  A unit is 64 columns (or all
// 16 or 32); several k-steps go with one unit, so that no operand row is
// transformed twice.
constexpr int kPwMaxC = 256;
PNN_HD constexpr int pw_unit_cols(int ncols) { return ncols % 64 == 0 ? 64 : ncols; }
inline bool pw_ok(int k, int stride, int ch, int ncols) {
  return k == 1 && stride == 1 && (ch == 16 || ch == 32 || (ch % 64 == 0 && ch <= kPwMaxC)) &&
         (ncols == 16 || ncols == 32 || ncols % 64 == 0) && (ch <= 64 || ncols <= 64);
}
constexpr int pw_raw_bytes(int ch, int esz) { return (kTcBM * (ch < 64 ? ch : 64) * esz + 1023) & ~1023; }
constexpr int pw_x_bytes(int ncols) { return kTcBM * pw_unit_cols(ncols) * 2; }
// units of an item: all of an m-tile's (its rows are transformed once), unless
// the launch has too few m-tiles to occupy the SMs twice over
inline int pw_item_units(int ncols, int64_t launch_mtiles) {
  return launch_mtiles >= 2 * (int64_t)device_sm_count() ? ncols / pw_unit_cols(ncols) : 1;
}
// 3x3 stride-1 forward / data gradient of k_c3_conv.cu (variant 5): ch channels
// of the A source, ncols GEMM columns in blocks of 64 (or all 16 or 32).  What an
// M tile is: a patch of 8 x 16 pixels, two whole 8 x 8 images, or 128 / (H W)
// whole smaller images (H and W powers of two).
struct C3Slots {
  int raw, op, wt, x;  // bytes of a raw, an operand and a weight slot, and of the second operand
  // small images or several column blocks somewhere in the launch: the general
  // form of the kernel (a forward of 16 channels takes 73 us with it, 60 with
  // the other, which has registers to spare)
  int any;
};
enum { C3_NONE = 0, C3_PATCH, C3_WHOLE, C3_SMALL };
PNN_HD inline int c3_kind(int H, int W) {
  if (H == 8 && W == 8) return C3_WHOLE;
  if (W % 8 == 0 && H % 16 == 0) return C3_PATCH;
  return H * W <= 32 && (H & (H - 1)) == 0 && (W & (W - 1)) == 0 ? C3_SMALL : C3_NONE;
}
// raw pixels of a k-step; bytes of an operand plane: a halo of 10 x 18 pixels,
// three copies of 10 x 16, or nine copies of 128 pixels (the latter two and four
// pixels that spread the two planes' stores over the banks)
PNN_HD constexpr int c3_raw_px(int kind) { return kind == C3_PATCH ? 180 : 128; }
PNN_HD constexpr int c3_plane(int kind) { return (kind == C3_PATCH ? 180 : kind == C3_WHOLE ? 484 : 1156) * 16; }
PNN_HD inline int c3_block(int ncols) { return ncols < 64 ? ncols : 64; }
PNN_HD constexpr int c3_wt_bytes(int block) { return 9 * block * 32; }  // 16 channels, nine taps
inline bool c3_ok(int k, int stride, int H, int W, int ch, int ncols) {
  auto cols = [](int c) { return c == 16 || c == 32 || (c > 0 && c % 64 == 0); };
  return k == 3 && stride == 1 && c3_kind(H, W) != C3_NONE && cols(ch) && cols(ncols);
}
inline void c3_add(C3Slots& s, int H, int W, int ncols, int esz, bool x) {
  const int kind = c3_kind(H, W), block = c3_block(ncols);
  auto most = [](int& a, int b) { if (a < b) a = b; };
  most(s.raw, c3_raw_px(kind) * 16 * esz);
  most(s.op, 2 * c3_plane(kind));
  most(s.wt, (c3_wt_bytes(block) + 1023) & ~1023);
  if (x) most(s.x, kTcBM * block * 2);
  if (kind == C3_SMALL || ncols > block) s.any = 1;
}
// Weight gradient of k_wg_conv.cu (a network's variant 4: 1x1, 5: 3x3): the geometry of one instance's
// k-steps.  1x1: kp pixels; 3x3: krows whole image rows (kp pixels) with the
// activation rows above and below.  Raw slot: x rows, then dY rows; operand
// slot: the M side's planes (8 channels each, apitch bytes), then (boff) the N
// side's.  A plane pitch of 8 / planes (mod 8) 16-byte rows spreads a warp's
// stores over the banks.
struct WgPlan {
  int kp, krows, lgw;
  int small;               // 3x3, whole images of at most 32 pixels: the N side holds a copy a tap
  int xch, ych, xrows;     // x and dY channels of a tile and raw rows of a k-step
  int x_is_a, mch, nch;    // M side: x or dY; channels of both sides (3x3: the N side holds three copies)
  int apitch, bpitch, boff;
  int yoff, raw, op;
};
constexpr int kWgRawMax = 40 * 1024;  // a raw slot: two stages and two operand slots fit
PNN_HD inline int wg_plane_pad(int ch) { return ch >= 64 ? 1 : 64 / ch; }
PNN_HD inline WgPlan wg_plan(int ks, int C, int K, int H, int W, bool xbf) {
  WgPlan p{};
  const int esz = xbf ? 2 : 4;
  if (ks == 1) {
    p.kp = 128;
    while (p.kp > 32 && p.kp * (C * esz + K * 4) > kWgRawMax) p.kp >>= 1;
    p.xch = C;
    p.ych = K;
    p.xrows = p.kp;
    p.x_is_a = C > K;
    p.mch = C > K ? C : K;
    p.nch = C > K ? K : C;
    p.bpitch = (p.kp + wg_plane_pad(p.nch)) * 16;
  } else {
    p.xch = C < 32 ? C : 32;
    p.ych = K < 128 ? K : 128;
    p.mch = p.ych;
    p.nch = p.xch;
    p.small = c3_kind(H, W) == C3_SMALL;
    while (1 << p.lgw < W) ++p.lgw;
    if (p.small) {
      p.kp = p.xrows = 64;
    } else {
      for (int r = 128 / W; r >= 1; --r) {
        if (H % r || (r * W) % 16 || (r + 2) * W > 256) continue;
        if ((r + 2) * W * p.xch * esz + r * W * p.ych * 4 > kWgRawMax) continue;
        p.krows = r;
        break;
      }
      p.kp = p.krows * W;
      p.xrows = (p.krows + 2) * W;  // (a multiple of 8)
    }
    p.bpitch = (p.xrows + wg_plane_pad(p.xch)) * 16;
  }
  p.apitch = (p.kp + wg_plane_pad(p.mch)) * 16;
  p.boff = p.mch / 8 * p.apitch;
  p.op = (p.boff + (ks == 1 ? 1 : p.small ? 9 : 3) * (p.nch / 8) * p.bpitch + 1023) & ~1023;
  p.yoff = (p.xrows * p.xch * esz + 127) & ~127;
  p.raw = (p.yoff + p.kp * p.ych * 4 + 1023) & ~1023;
  return p;
}
bool wg_fits(int raw_bytes, int op_bytes);
inline bool wg_ok(int k, int stride, int C, int K, int H, int W, bool xbf) {
  auto pow2 = [](int v, int lo, int hi) { return v >= lo && v <= hi && (v & (v - 1)) == 0; };
  if (stride != 1) return false;
  if (k == 1) {
    if (!pow2(C, 16, 256) || !pow2(K, 16, 256) || (C > 64 && K > 64)) return false;
  } else {
    // blocks of 32 x 128 channels, or all of a narrower layer's
    if (k != 3 || (C != 16 && (C <= 0 || C % 32 != 0)) || (!pow2(K, 16, 128) && (K <= 0 || K % 128 != 0))) return false;
    if (c3_kind(H, W) != C3_SMALL && !pow2(W, 8, 32)) return false;
  }
  const WgPlan p = wg_plan(k, C, K, H, W, xbf);
  return p.kp > 0 && wg_fits(p.raw, p.op);
}
// tiles of an instance per split: blocks of x channels and of dY channels
PNN_HD inline int wg_xblocks(int ks, int C) { return ks == 3 && C > 32 ? C / 32 : 1; }
PNN_HD inline int wg_ntiles(int ks, int C, int K) { return wg_xblocks(ks, C) * (ks == 3 && K > 128 ? K / 128 : 1); }
// whether a layer needs the general form of the 3x3 kernel
inline bool wg_any(int ks, int H, int W, int K) { return ks == 3 && (c3_kind(H, W) == C3_SMALL || K > 128); }
// Splits of the instances of one launch: about two tiles per SM over the
// launch, each instance in proportion to the bytes it moves, whole k-steps.
// (With 2 x SMs splits for every instance, as a launch of its own needs, eight
// instances wrote and reduced eight times the partial sums.)
struct WgSplit { int splits, pix; };
inline WgSplit wg_split(int64_t rows, int kp, int ntiles, double bytes, double launch_bytes) {
  const double share = 2.0 * device_sm_count() * bytes / launch_bytes / ntiles;
  int64_t s = (int64_t)(share + 0.5);
  const int64_t steps = (rows + kp - 1) / kp;
  s = s < 1 ? 1 : (s > steps ? steps : s);
  // k-steps a split: at least 256 pixels (a partial sum is as large as the layer)
  const int64_t per = std::max<int64_t>((steps + s - 1) / s, (256 + kp - 1) / kp);
  return WgSplit{(int)((steps + per - 1) / per), (int)(per * kp)};
}
// N columns of a tile when the layer needs several: 128 for the TMA-fed
// forward and data gradient (a smaller operand slot leaves room for more
// pipeline stages), 256 otherwise.
inline int tc_ntile_cols(int mode, int variant) { return variant == 1 && mode != 2 ? 128 : 256; }
// M rows of a tile: 256 for the TMA-fed weight gradient of a layer with at
// most 128 input channels (two MMA halves share each B operand, so a layer
// with up to 256 (r,s,c) rows makes one pass over the pixels; a tile then
// holds whole taps, all inside the activation box), 128 otherwise.
inline int tc_tile_rows(int mode, int variant, int C) { return mode == 2 && variant == 1 && C <= 128 ? 256 : kTcBM; }
// 2-D tensor map (CUtensorMap, 128 bytes at `map`) over rows x inner elements
// (bf16 or fp32, row pitch inner * element size) with box
// [box_rows][box_inner]; swz: swizzle span in bytes (128, 64, 32 or 0).
// Returns 0, or non-zero with a message in *why.
// general form: dims, byte strides of dims 1 .., box, innermost first; rank 2 to 4
int encode_tensor_map_nd(void* map, const void* base, bool bf16, int rank, const int64_t* dims, const int64_t* strides,
                         const int* box, int swz, const char** why);
// [images][H][W][C] with a box of box_c channels x box_w x box_h x box_n
int encode_tensor_map_nhwc(void* map, const void* base, bool bf16, int C, int W, int H, int B, int box_c, int box_w,
                           int box_h, int box_n, int swz, const char** why);
// the maps (a, unused, output, second operand; 128 bytes apart) of a k_c3_conv.cu instance
int encode_c3_maps(void* maps, bool fwd, const void* a, bool a_bf16, int ch, void* out, int ncols,
                   const void* x, int B, int H, int W, const char** why);
int encode_tensor_map_2d(void* map, const void* base, bool bf16, int64_t inner, int64_t rows, int box_inner,
                         int box_rows, int swz, const char** why);

constexpr int kBnbRowsPerTile = 256;  // BN backward reduce/apply tiles: at most this many rows of a wide layer
// rows of a BN-backward tile of M rows x C channels: about 32K elements a CTA; a
// layer with few rows gets 16 tiles, of at least 2K elements (a batch of 8 at 32 x
// 32 x 16 had 4 tiles, the 512 x 512 gradient of VGG-16's last layer 2).  More do
// not pay: a launch holds several instances, and every CTA loads seven parameters a
// channel (two tiles an SM for each instance: ResNet-1001 with 4 subnetworks 26.6 ->
// 28.8 ms; 32 tiles: 26.5 -> 26.7).  (bnb_fixed_rows: the reduction of an fp32
// network, see "Fixed order" in k_simt.cu.)
inline int bnb_fixed_rows(int C) { return C > 0 && 32768 / C > kBnbRowsPerTile ? 32768 / C : kBnbRowsPerTile; }
inline int bnb_rows_per_tile(int C, int64_t M) {
  int rows = bnb_fixed_rows(C);
  while (rows > 8 && (int64_t)rows * C > 2048 && M < 16 * (int64_t)rows) rows /= 2;
  return rows;
}
// The TMA-fed weight gradient loads a k-step's activation rows for all taps
// as one halo box and the output-gradient rows as another: channels 8..64
// (dividing 64) or multiples of 128 up to 512, at most 128 output channels
// (one N tile), a halo of at most 256 rows, and two stages in shared memory.
inline bool tma_wgrad_ok(int k, int stride, int pad, int C, int K, int W, bool xbf) {
  if (!(stride == 1 && ((k == 1 && pad == 0) || (k == 3 && pad == 1)))) return false;
  if (!(C % 8 == 0 && ((C <= 64 && 64 % C == 0) || (C % 128 == 0 && C <= 512)))) return false;
  if (K % 8 != 0 || K > 128) return false;
  const WgBoxes b = wg_boxes(C, K, W, pad, xbf);
  return b.hrows <= 256 && conv_tma_fits(2, 128, wg_raw_bytes(b));
}
// CUDA-core forward and data gradient: 64 x 64, 128 x 32 or 64 x 16 tiles by
// the GEMM's columns (16: a batch of 8 still gives every SM a tile); forward
// only: variant 3, at most 32 taps x channels (the 3-channel stem and C^j
// convs), one thread a pixel; variant 4, 64 x 16 tiles of an fp32 network in
// clusters of four, which form one partial of the BN statistics.
struct ConvTile { int BM, BN; };
inline ConvTile simt_tile(int variant) {
  return variant == 0                   ? ConvTile{64, 64}
         : variant == 1                 ? ConvTile{128, 32}
         : variant == 2 || variant == 4 ? ConvTile{64, 16}
                                        : ConvTile{256, 16};
}
inline int simt_variant(int ncols) { return ncols <= 16 ? 2 : (ncols <= 32 ? 1 : 0); }
inline int simt_fwd_variant(int k, int C, int K, bool fp32) {
  const int v = k * k * C <= 32 && C < 8 ? 3 : simt_variant(K);
  return fp32 && v == 2 ? 4 : v;
}
constexpr int kQuad = 4;  // CTAs of a cluster of variant 4
inline int simt_fwd_mtiles(int variant, int64_t M) {
  const int bm = simt_tile(variant).BM, group = variant == 4 ? kQuad : 1;
  return (int)((M + bm * group - 1) / (bm * group)) * group;
}
// rows of a partial of the BN statistics: the kernel's tile, or, of an fp32
// network, fixed by the layer's width ("Fixed order", k_simt.cu)
inline int simt_stat_rows(int variant, int K, bool fp32) {
  return !fp32 ? simt_tile(variant).BM : K <= 16 ? 256 : K <= 32 ? 128 : 64;
}
// CUDA-core weight gradient: 64 or 16 output channels a tile (0, 1), few input
// channels with at most 16 (2) or more (3) output channels, 1x1 stride 1 with at
// most 4 input channels (4).  An fp32 network takes 0 and 1, which add a split's
// pixels one after another.
inline int simt_wgrad_variant(int k, int stride, int C, int K, bool fp32) {
  if (fp32) return K <= 16 ? 1 : 0;
  if (k == 1 && stride == 1 && C <= 4) return 4;
  return k * k * C <= 32 && C < 8 ? (K <= 16 ? 2 : 3) : (K <= 16 ? 1 : 0);
}
inline int simt_wgrad_rows(int variant) { return variant == 1 ? 16 : 64; }
// CTAs an SM that the splits of a CUDA-core weight gradient aim at (the
// few-channel kernels' partial sums are small)
inline int simt_wgrad_ctas(int variant) { return variant >= 2 ? 8 : 2; }
constexpr int kWgradBM = 64, kWgradBN = 64, kWgradBK = 16;

}  // namespace pnn
