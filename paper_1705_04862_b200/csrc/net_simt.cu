// The network's layers as contractions on the CUDA cores (float accumulate):
// forward with fused bias + ReLU, data gradients with the ReLU mask of the layer
// below fused, weight gradients as split-k partial sums reduced in a fixed order.
#include "gemm_ffma.cuh"
#include "gemm_tc3.cuh"
#include "kernels.h"

namespace paac {

static int pick_splits(int M, int N, int K) {
  const int blocks = ((M + 63) / 64) * ((N + 63) / 64);
  int s = (592 + blocks - 1) / blocks;
  const int by_k = (K + 127) / 128;
  if (s > by_k) s = by_k;
  if (s > 512) s = 512;
  if (s < 1) s = 1;
  return gemm_k_splits(K, s);
}

// Shapes of the CUDA-core contraction for N columns (16, 32, or 64 and more).  At 128 states forward and 640 backward (where
// nothing goes to the tensor cores, see below) the larger network's layers run at 9 to 14 and 13 to 20 TMAC/s of the 36 the multiply-add pipe
// could do, with 54 to 65 and 58 to 82 % of the issue slots busy.  The wide shape (8 x 8 per lane for 64 columns, 8 x 4 below, where 8 x 8 leaves tiles of too
// many rows) wins from two warps per scheduler on (1184 of them; 19.8 against 18.4 TMAC/s for the fully connected layer's
// weight gradient), below that 4 x 4 (18.4 against 12.2 with one and a half), and 2 x 4 where even that leaves a scheduler
// without a warp (592).  4 x 4 with 64 columns comes in blocks of two warps: the
// second layer's 10368 rows then fill the device in more even rounds (34 -> 30 us, the third layer's 6272 the same).
constexpr int FF_SMS = 148;

// ---- which contractions go to the tensor cores ----
// Splits of k for an M x N result there: two blocks per SM, four blocks of k and more to each.
static int t3_splits(int M, int N, int K) {
  const int bn = N < 64 ? N : 64, tiles = (M + T3_BM - 1) / T3_BM * ((N + bn - 1) / bn);
  int s = 2 * FF_SMS / tiles;
  const int by_k = K / (4 * T3_BK);
  if (s > by_k) s = by_k;
  return s < 1 ? 1 : gemm_k_splits(K, s, T3_BK);
}
// By itself only where its error against sums in 64 bits is no larger, in the 2-norm, than that of the multiply-adds' chain, measured
// over both networks, 20 to 960 rows, before and after training.  (The pieces have 22 of a float's 24 bits.  That shows in elements with few
// terms: root mean square of the error over the sum of the terms' sizes 0.5 to 1.1 times the chain's in data gradients, 0.5 to 1.6 times in
// weight gradients.  Who wants chains throughout sets PAAC_OPT_CUDA_CORES_ONLY.)
// Data gradients, M rows.  A tile takes about a microsecond per block of 32 k, whatever the number of tiles up to two per SM, where the
// CUDA cores take time with the multiply-adds: 11 M of them per block and 80 M in all is where the two meet.  (us, CUDA cores / tensor cores,
// larger network: third layer, 18 blocks, 40 states 25 / 26, 64 states 29 / 25, 640 states 105 / 54; second layer, 8 blocks, 40 states 19 / 19, 80 states
// 26 / 19, 640 states 126 / 67; fully connected layer, 16 blocks, 80 states 19 / 23, 120 states 25 / 23, 640 states 70 / 29.)  Errors,
// 2-norm: 1.2 to 1.5e-7 instead of 1.3 to 2.9e-7, 0.5 to 0.95 times the chain's.
// The forward pass stays on the CUDA cores, whose chains of multiply-adds are the same for every batch: sums as exact but in another order put
// a unit or two per pass on the other side of the ReLU, and training then runs apart from there.
template <class T> static bool t3_allowed(const LaunchCtx& lc) { return !lc.cuda_cores_only && lc.error_word != nullptr && (sizeof(T) == 4 || lc.bf16_sums_on_tensor_cores); }
template <class T> static bool t3_pays(const LaunchCtx& lc, long long M, int N, int K) {
  if (lc.fp32_tensor_cores) return lc.error_word != nullptr;
  const long long blocks = (K + T3_BK - 1) / T3_BK, macs = M * N * K;
  return t3_allowed<T>(lc) && macs >= blocks * 11000000 && macs >= 80000000;
}
// Weight gradients, whose k is split until the device is full: from 64 M multiply-adds on (first layer of the smaller network, 40 states 14 / 11 us,
// 160 states 31 / 20, 960 states 152 / 66; second layer 80 states 13 / 11, 640 states 43 / 20), and from as many rows on that the sums, not the operands,
// make the error: 2-norm of a convolution's 0.2 to 0.95 times the chain's from 2048 rows on (40 states of the third layer, 1960 rows: 1.03
// times), of the fully connected layer's 0.5 to 0.99 times from 512 on, in either storage (268 to 511 rows: 0.5 to 1.33 times).
template <class T, class LA> static bool t3_wgrad_pays(const LaunchCtx& lc, int J, int CO, int K) {
  if (lc.fp32_tensor_cores) return lc.error_word != nullptr;
  constexpr int LEAST = T3Table<LA>::use ? 2048 : 512;      // of a convolution's windows, or of the fully connected layer
  return t3_allowed<T>(lc) && K >= LEAST && (long long)J * CO * K >= 64000000;
}
static size_t ff_heads_scratch_floats(const NetDims& nd, int n);
static int ff_shape(int N, long long outputs) {              // outputs of all classes and splits
  if (outputs >= 1184LL * 32 * 8 * (N >= 64 ? 8 : 4)) return 2;
  return outputs >= 592LL * 32 * 16 ? 1 : 0;
}
template <int N, int SHAPE, class LA, class LB, class EP>
static void ff_launch(LaunchCtx& lc, int kid, int M, int n_cols, int K, int kps, int classes, LA la, LB lb, EP ep) {
  constexpr int WIDE_BK = sizeof(typename LA::Elem) == 1 ? 32 : 16;       // bytes pass through registers, one block ahead
  if constexpr (N == 16) {
    if constexpr (SHAPE == 2) gemm_ffma<8, 8, 4, 4, 1, WIDE_BK>(lc, kid, M, n_cols, K, kps, classes, la, lb, ep);
    else if constexpr (SHAPE == 1) gemm_ffma<8, 4, 4, 4, 1, 32>(lc, kid, M, n_cols, K, kps, classes, la, lb, ep);
    else gemm_ffma<8, 2, 4, 4, 1, 64>(lc, kid, M, n_cols, K, kps, classes, la, lb, ep);
  } else if constexpr (N == 32) {
    if constexpr (SHAPE == 2) gemm_ffma<4, 8, 4, 4, 1, WIDE_BK>(lc, kid, M, n_cols, K, kps, classes, la, lb, ep);
    else if constexpr (SHAPE == 1) gemm_ffma<4, 4, 4, 4, 1, 32>(lc, kid, M, n_cols, K, kps, classes, la, lb, ep);
    else gemm_ffma<4, 2, 4, 4, 1, 64>(lc, kid, M, n_cols, K, kps, classes, la, lb, ep);
  } else {
    if constexpr (SHAPE == 2) gemm_ffma<4, 8, 8, 4, 1, 16>(lc, kid, M, n_cols, K, kps, classes, la, lb, ep);
    else if constexpr (SHAPE == 1) gemm_ffma<4, 4, 4, 1, 2, 32>(lc, kid, M, n_cols, K, kps, classes, la, lb, ep);
    else gemm_ffma<4, 2, 4, 2, 2, 64>(lc, kid, M, n_cols, K, kps, classes, la, lb, ep);
  }
}
template <int N, class LA, class LB, class EP>
static void ff_rows(LaunchCtx& lc, int kid, int M, int n_cols, int K, int kps, int classes, LA la, LB lb, EP ep) {
  const int shape = ff_shape(N, (long long)M * n_cols * classes * ((K + kps - 1) / kps));
  if (shape == 2) ff_launch<N, 2>(lc, kid, M, n_cols, K, kps, classes, la, lb, ep);
  else if (shape == 1) ff_launch<N, 1>(lc, kid, M, n_cols, K, kps, classes, la, lb, ep);
  else ff_launch<N, 0>(lc, kid, M, n_cols, K, kps, classes, la, lb, ep);
}

// Weight gradients: C(j, co) = sum over output positions of window(j) * gradient(co), one run of positions per split;
// the splits' sums (and the bias gradient's, the column sums of the second operand) are added, in split order, by
// finish_gradients().
struct FfWgradPlan { int splits, kps; size_t part, total; };      // floats: the weights' partial sums, and all of them
static FfWgradPlan ff_wgrad_plan(int J, int CO, int K, bool tensor) {
  FfWgradPlan p;
  p.splits = tensor ? t3_splits(J, CO, K) : pick_splits(CO, J + 1, K);
  p.kps = gemm_k_per_split(K, p.splits, tensor ? T3_BK : 16);
  p.part = (size_t)p.splits * J * CO;
  p.total = (p.part + (size_t)p.splits * CO + 63) / 64 * 64;
  return p;
}
template <int CO_TILE, class LA, class LB>
static void ff_wgrad(LaunchCtx& lc, int kid, int J, int CO, int K, LA window, LB grad_rows, float scale, float* gw, float* gb,
                     float* scratch, GradSegments* segs) {
  typedef typename LB::Elem T;
  const bool tensor = t3_wgrad_pays<T, LA>(lc, J, CO, K);
  const FfWgradPlan p = ff_wgrad_plan(J, CO, K, tensor);
  FfPartialColsum ep;
  ep.part = scratch; ep.M = J; ep.N = CO; ep.colpart = scratch + p.part;
  // 64 x 64 tiles of 8 x 8 per lane where they give every SM three blocks, 128 x 32 of 8 x 4 where those give it one
  if (tensor)
    gemm_tc3<CO_TILE>(lc, kid, J, CO, K, p.kps, 1, window, grad_rows, ep);
  else if (CO_TILE == 64 && (J + 63) / 64 * ((CO + 63) / 64) * p.splits >= 3 * FF_SMS)
    gemm_ffma<4, 8, 8, 2, 1, 16>(lc, kid, J, CO, K, p.kps, 1, window, grad_rows, ep);
  else if (CO_TILE == 32 && (J + 127) / 128 * p.splits >= FF_SMS)
    gemm_ffma<4, 8, 4, 4, 1, 16>(lc, kid, J, CO, K, p.kps, 1, window, grad_rows, ep);
  else
    ff_rows<CO_TILE>(lc, kid, J, CO, K, p.kps, 1, window, grad_rows, ep);
  if (!add_grad_segment(segs, scratch, gw, p.splits, J, CO, scale, !tensor) || !add_grad_segment(segs, ep.colpart, gb, p.splits, 1, CO, 1.f, !tensor))
    lc.host_failure = true;
}

template <class G, class TIn, class T, class TW>
static void conv_fwd(LaunchCtx& lc, int kid, const TIn* x, const TW* w, const float* bias, T* out, int n,
                     float scale) {
  const int M = n * G::OH * G::OW;
  const FfWindow<G, TIn> window{x};
  const FfRows<TW> weights{w, G::KK};
  const FfBiasRelu<T> ep{out, bias, G::CO, scale};
  if (lc.fp32_tensor_cores) gemm_tc3<G::CO>(lc, kid, M, G::CO, G::KK, G::KK, 1, window, weights, ep);
  else ff_rows<G::CO>(lc, kid, M, G::CO, G::KK, G::KK, 1, window, weights, ep);
}
// With few states the fully connected layer is a handful of tiles over a reduction of thousands: the reduction is then
// split over many blocks (partial sums in scratch, added by launch_simt_tail) so that the weight matrix is streamed by
// the whole device instead of by four blocks.  Returns the number of splits left in scratch (0: the layer is complete).
template <class T, class TW>
static int fc_fwd(LaunchCtx& lc, int kid, const T* x, const TW* w, const float* bias, T* out, int n,
                   int IN, int F, float* scratch) {
  const bool tensor = lc.fp32_tensor_cores;
  const int splits = tensor ? t3_splits(n, F, IN) : pick_splits(n, F, IN);
  const int kps = splits <= 1 ? IN : gemm_k_per_split(IN, splits, tensor ? T3_BK : 16);
  auto launch = [&](auto ep) {
    if (tensor) gemm_tc3<64>(lc, kid, n, F, IN, kps, 1, FfRows<T>{x, IN}, FfRows<TW>{w, IN}, ep);
    else ff_rows<64>(lc, kid, n, F, IN, kps, 1, FfRows<T>{x, IN}, FfRows<TW>{w, IN}, ep);
  };
  if (splits <= 1) launch(FfBiasRelu<T>{out, bias, F, 1.f});
  else launch(FfPartial{scratch, n, F});
  return splits <= 1 ? 0 : splits;
}
template <class G, class T, class TW>
static void conv_dgrad(LaunchCtx& lc, int kid, const T* g, const TW* w, const T* act_in, T* gin, int n) {
  if constexpr (G::S == 2 && G::K == 4 && G::H % 2 == 0 && G::W % 2 == 0) {
    // four parity classes, each a dense contraction over its own four taps (a quarter of the multiply-adds)
    const int M = n * (G::H / 2) * (G::W / 2), K = 4 * G::CO;
    const FfDgradClass<G, T> rows{g};
    const FfWeightClass<G, TW> weights{w, 0};
    const FfReluMaskClass<G, T> ep{gin, act_in, 0};
    if (t3_pays<T>(lc, M, 4 * G::C, K))
      gemm_tc3<64>(lc, kid, M, 4 * G::C, K, K, 1, rows, T3WeightClasses<G, TW>{w}, T3ReluMaskClasses<G, T>{gin, act_in});
    else
      ff_rows<G::C>(lc, kid, M, G::C, K, K, 4, rows, weights, ep);
  } else {
    const int M = n * G::H * G::W, K = G::K * G::K * G::CO;
    const FfDgradWindow<G, T> rows{g};
    const FfWeightT<G, TW> weights{w};
    const FfReluMask<T> ep{gin, act_in, G::C};
    if (t3_pays<T>(lc, M, G::C, K)) gemm_tc3<G::C>(lc, kid, M, G::C, K, K, 1, rows, weights, ep);
    else ff_rows<G::C>(lc, kid, M, G::C, K, K, 1, rows, weights, ep);
  }
}
template <class G, class TIn, class T>
static void conv_wgrad(LaunchCtx& lc, int kid, const T* g, const TIn* x, int n, float scale, float* gw,
                       float* gb, float* scratch, GradSegments* segs) {
  ff_wgrad<G::CO>(lc, kid, G::KK, G::CO, n * G::OH * G::OW, FfWindowT<G, TIn>{x}, FfCols<T>{g, G::CO}, scale, gw, gb, scratch, segs);
}
template <class T, class TW>
static void fc_dgrad(LaunchCtx& lc, int kid, const T* g, const TW* w, const T* act_in, T* gin, int n,
                     int IN, int F) {
  const FfReluMask<T> ep{gin, act_in, IN};
  if (t3_pays<T>(lc, n, IN, F)) gemm_tc3<64>(lc, kid, n, IN, F, F, 1, FfRows<T>{g, F}, FfCols<TW>{w, IN}, ep);
  else ff_rows<64>(lc, kid, n, IN, F, F, 1, FfRows<T>{g, F}, FfCols<TW>{w, IN}, ep);
}
template <class T>
static void fc_wgrad(LaunchCtx& lc, int kid, const T* g, const T* x, int n, int IN, int F, float* gw,
                     float* gb, float* scratch, GradSegments* segs) {
  ff_wgrad<64>(lc, kid, IN, F, n, FfCols<T>{x, IN}, FfCols<T>{g, F}, 1.f, gw, gb, scratch, segs);
}

template <class T, class TW>
static int forward_t(LaunchCtx& lc, int arch, const NetDims& nd, const float* theta, const TW* w,
                      const uint8_t* frames, int n, void* const act[], float* scratch) {
  const LayerDims* d = nd.layer;
  const float s255 = 1.0f / 255.0f;
  if (arch == PAAC_ARCH_NIPS) {
    conv_fwd<NipsConv1, uint8_t, T, TW>(lc, KID_CONV1_FWD, frames, w + d[0].w_off, theta + d[0].b_off, (T*)act[0], n, s255);
    conv_fwd<NipsConv2, T, T, TW>(lc, KID_CONV2_FWD, (const T*)act[0], w + d[1].w_off, theta + d[1].b_off, (T*)act[1], n, 1.f);
    return fc_fwd<T, TW>(lc, KID_FC_FWD, (const T*)act[1], w + d[2].w_off, theta + d[2].b_off, (T*)act[2], n, 2592, 256, scratch);
  } else {
    conv_fwd<NatConv1, uint8_t, T, TW>(lc, KID_CONV1_FWD, frames, w + d[0].w_off, theta + d[0].b_off, (T*)act[0], n, s255);
    conv_fwd<NatConv2, T, T, TW>(lc, KID_CONV2_FWD, (const T*)act[0], w + d[1].w_off, theta + d[1].b_off, (T*)act[1], n, 1.f);
    conv_fwd<NatConv3, T, T, TW>(lc, KID_CONV3_FWD, (const T*)act[1], w + d[2].w_off, theta + d[2].b_off, (T*)act[2], n, 1.f);
    return fc_fwd<T, TW>(lc, KID_FC_FWD, (const T*)act[2], w + d[3].w_off, theta + d[3].b_off, (T*)act[3], n, 3136, 512, scratch);
  }
}

// one layer of the backward pass: its weight gradient and/or the data gradient handed to the layer below
template <class T, class TW>
static void backward_layer_t(LaunchCtx& lc, int arch, const NetDims& nd, const TW* w, const uint8_t* frames, int n,
                             void* const act[], void* const gact[], float* grad, float* scratch, GradSegments* segs, int l,
                             bool wg, bool dg) {
  const LayerDims* d = nd.layer;
  const float s255 = 1.0f / 255.0f;
  const T* g = (const T*)gact[l];
  const T* x = l > 0 ? (const T*)act[l - 1] : nullptr;
  T* gin = l > 0 ? (T*)gact[l - 1] : nullptr;
  float* gw = grad + d[l].w_off; float* gb = grad + d[l].b_off;
  const TW* wl = w + d[l].w_off;
  if (arch == PAAC_ARCH_NIPS) {
    if (l == 2) {
      if (wg) fc_wgrad<T>(lc, KID_FC_WGRAD, g, x, n, 2592, 256, gw, gb, scratch, segs);
      if (dg) fc_dgrad<T, TW>(lc, KID_FC_DGRAD, g, wl, x, gin, n, 2592, 256);
    } else if (l == 1) {
      if (wg) conv_wgrad<NipsConv2, T, T>(lc, KID_CONV2_WGRAD, g, x, n, 1.f, gw, gb, scratch, segs);
      if (dg) conv_dgrad<NipsConv2, T, TW>(lc, KID_CONV2_DGRAD, g, wl, x, gin, n);
    } else if (wg) {
      conv_wgrad<NipsConv1, uint8_t, T>(lc, KID_CONV1_WGRAD, g, frames, n, s255, gw, gb, scratch, segs);
    }
  } else {
    if (l == 3) {
      if (wg) fc_wgrad<T>(lc, KID_FC_WGRAD, g, x, n, 3136, 512, gw, gb, scratch, segs);
      if (dg) fc_dgrad<T, TW>(lc, KID_FC_DGRAD, g, wl, x, gin, n, 3136, 512);
    } else if (l == 2) {
      if (wg) conv_wgrad<NatConv3, T, T>(lc, KID_CONV3_WGRAD, g, x, n, 1.f, gw, gb, scratch, segs);
      if (dg) conv_dgrad<NatConv3, T, TW>(lc, KID_CONV3_DGRAD, g, wl, x, gin, n);
    } else if (l == 1) {
      if (wg) conv_wgrad<NatConv2, T, T>(lc, KID_CONV2_WGRAD, g, x, n, 1.f, gw, gb, scratch, segs);
      if (dg) conv_dgrad<NatConv2, T, TW>(lc, KID_CONV2_DGRAD, g, wl, x, gin, n);
    } else if (wg) {
      conv_wgrad<NatConv1, uint8_t, T>(lc, KID_CONV1_WGRAD, g, frames, n, s255, gw, gb, scratch, segs);
    }
  }
}

// Where layer l's partial sums start in the update's scratch; l = number of layers: the heads' region; one more: the end.
// Every layer has a region of its own, large enough for either contraction: partial sums stay until finish_gradients() has run.
static size_t ff_scratch_offset(const NetDims& nd, int n, int l) {
  size_t off = 0;
  for (int q = 0; q < l && q <= nd.n_conv; ++q) {
    const LayerDims& d = nd.layer[q];
    const int J = q < nd.n_conv ? d.K * d.K * d.C : d.H * d.W * d.C, K = n * d.OH * d.OW;
    const size_t cuda = ff_wgrad_plan(J, d.CO, K, false).total, tensor = ff_wgrad_plan(J, d.CO, K, true).total;
    off += cuda > tensor ? cuda : tensor;
  }
  if (l > nd.n_conv + 1) off += ff_heads_scratch_floats(nd, n);
  return off;
}

void simt_backward_layer(LaunchCtx& lc, int arch, int prec, const NetDims& nd, const float* theta, const bf16* theta16,
                         const uint8_t* frames, int n, void* const act[], void* const gact[], float* grad,
                         float* scratch, GradSegments* segs, int layer, bool wgrad, bool dgrad) {
  float* sc = scratch + ff_scratch_offset(nd, n, layer);
  if (prec == PAAC_BF16)
    backward_layer_t<bf16, bf16>(lc, arch, nd, theta16, frames, n, act, gact, grad, sc, segs, layer, wgrad, dgrad);
  else
    backward_layer_t<float, float>(lc, arch, nd, theta, frames, n, act, gact, grad, sc, segs, layer, wgrad, dgrad);
}

int simt_forward(LaunchCtx& lc, int arch, int prec, const NetDims& nd, const float* theta,
                 const bf16* theta16, const uint8_t* frames, int n, void* const act[], float* scratch) {
  if (prec == PAAC_BF16) return forward_t<bf16, bf16>(lc, arch, nd, theta, theta16, frames, n, act, scratch);
  return forward_t<float, float>(lc, arch, nd, theta, theta, frames, n, act, scratch);
}

size_t simt_scratch_floats(int arch, const NetDims& nd, int n, int n_fwd) {
  (void)arch;
  const size_t best = ff_scratch_offset(nd, n, nd.n_conv + 2);      // all of an update's partial sums
  // split-k partial sums of the fully connected layer's forward pass, which only ever sees n_fwd states at a time
  const LayerDims& f = nd.layer[nd.n_conv];
  const int IN = f.H * f.W * f.C;
  const int cuda = pick_splits(n_fwd, nd.F, IN), tensor = t3_splits(n_fwd, nd.F, IN);
  const size_t fwd = (size_t)(cuda > tensor ? cuda : tensor) * n_fwd * nd.F;
  return best > fwd ? best : fwd;
}

// ---- heads backward (tiny contractions over the A+1 head units) ------------------------------
// Both heads in one kernel, for either storage type and either hidden size (the tensor-core path has one of its own for
// 512 bf16 units): with dz[b][k] the loss gradient at output k of row b (the value is row k = A of the combined matrix),
//   g_fc[b][i] = (h[b][i] > 0) * sum_k dz[b][k] W[k][i],   dW[k][i] = sum_b dz[b][k] h[b][i],   db[k] = sum_b dz[b][k].
// A thread owns one hidden unit; its weights and gradient sums stay in registers, so a row costs it one load of h and
// 2 NK multiply-adds.  A block takes 64 units and the rows of one split (at most about 128), FH_ROWS at a time, the next
// ones on their way while these are used: a chain of some microseconds whatever the batch.
constexpr int FH_THREADS = 64;
template <class T, class TW, int NK>
__global__ void __launch_bounds__(FH_THREADS)
heads_backward_kernel(const T* h, const float* dz, const float* dV, const TW* wpi, const TW* wv, int n, int F, int A, int rows_per,
                      T* g_fc, float* part_w, float* part_b, float* part_vw, float* part_vb) {
  constexpr int FH_ROWS = NK <= 20 ? 32 : 16;
  __shared__ float dzs[FH_ROWS][NK];
  const int tid = threadIdx.x, col = blockIdx.y * FH_THREADS + tid;
  pdl_entry();
  float w[NK], acc[NK], accb = 0.f;
#pragma unroll
  for (int k = 0; k < NK; ++k) {
    acc[k] = 0.f;
    w[k] = k < A ? to_f(wpi[(size_t)k * F + col]) : (k == A ? to_f(wv[col]) : 0.f);
  }
  const int r0 = blockIdx.x * rows_per, r1 = min(n, r0 + rows_per);
  constexpr int DZ = (FH_ROWS * NK + FH_THREADS - 1) / FH_THREADS;
  float hv[FH_ROWS], dv[DZ];
  auto fetch = [&](int rb) {
#pragma unroll
    for (int j = 0; j < FH_ROWS; ++j) hv[j] = rb + j < r1 ? to_f(h[(size_t)(rb + j) * F + col]) : 0.f;
#pragma unroll
    for (int q = 0; q < DZ; ++q) {
      const int i = tid + q * FH_THREADS, r = rb + i / NK, k = i % NK;
      dv[q] = i < FH_ROWS * NK && r < r1 ? (k < A ? dz[(size_t)r * A + k] : (k == A ? dV[r] : 0.f)) : 0.f;
    }
  };
  fetch(r0);
  for (int rb = r0; rb < r1; rb += FH_ROWS) {
    float hc[FH_ROWS];
#pragma unroll
    for (int j = 0; j < FH_ROWS; ++j) hc[j] = hv[j];
    __syncthreads();
#pragma unroll
    for (int q = 0; q < DZ; ++q) {
      const int i = tid + q * FH_THREADS;
      if (i < FH_ROWS * NK) dzs[i / NK][i % NK] = dv[q];
    }
    __syncthreads();
    if (rb + FH_ROWS < r1) fetch(rb + FH_ROWS);
    if (tid <= A)
#pragma unroll
      for (int j = 0; j < FH_ROWS; ++j) accb += dzs[j][tid];          // rows past the end hold zeros
#pragma unroll
    for (int j = 0; j < FH_ROWS; ++j) {
      float g = 0.f;
#pragma unroll
      for (int k = 0; k < NK; ++k) {
        const float d = dzs[j][k];
        g = fmaf(d, w[k], g);
        acc[k] = fmaf(d, hc[j], acc[k]);
      }
      if (rb + j < r1) g_fc[(size_t)(rb + j) * F + col] = from_f<T>(hc[j] > 0.f ? g : 0.f);
    }
  }
  const size_t split = blockIdx.x;
#pragma unroll
  for (int k = 0; k < NK; ++k) {
    if (k < A) part_w[(split * A + k) * F + col] = acc[k];
    else if (k == A) part_vw[split * F + col] = acc[k];
  }
  if (blockIdx.y == 0) {
    if (tid < A) part_b[split * A + tid] = accb;
    else if (tid == A) part_vb[split] = accb;
  }
}
static size_t ff_heads_scratch_floats(const NetDims& nd, int n) {
  return (size_t)pick_splits(nd.A + 1, nd.F + 1, n) * (nd.A + 1) * (nd.F + 1) + 8;
}

template <class T, class TW>
static void heads_backward_t(LaunchCtx& lc, const NetDims& nd, const TW* w, const T* h, int n,
                             const float* dz, const float* dV, T* gact_fc, float* grad, float* scratch, GradSegments* segs) {
  const int A = nd.A, F = nd.F;
  const int splits = pick_splits(A + 1, F + 1, n), rows_per = gemm_k_per_split(n, splits);
  float* part_w = scratch + ff_scratch_offset(nd, n, nd.n_conv + 1);
  float* part_b = part_w + (size_t)splits * A * F;
  float* part_vw = part_b + (size_t)splits * A;
  float* part_vb = part_vw + (size_t)splits * F;
  auto launch = [&](auto kern) {
    KernelScope scope(lc, KID_HEADS_BWD);
    launch_kernel_overlapped(lc, kern, dim3(splits, F / FH_THREADS), dim3(FH_THREADS), 0, h, dz, dV, w + nd.pi_w, w + nd.v_w, n, F, A,
                             rows_per, gact_fc, part_w, part_b, part_vw, part_vb);
  };
  if (A < 8) launch(heads_backward_kernel<T, TW, 8>);
  else if (A < 20) launch(heads_backward_kernel<T, TW, 20>);
  else launch(heads_backward_kernel<T, TW, 33>);
  if (!add_grad_segment(segs, part_w, grad + nd.pi_w, splits, 1, F * A, 1.f, true) || !add_grad_segment(segs, part_b, grad + nd.pi_b, splits, 1, A, 1.f, true) ||
      !add_grad_segment(segs, part_vw, grad + nd.v_w, splits, 1, F, 1.f, true) || !add_grad_segment(segs, part_vb, grad + nd.v_b, splits, 1, 1, 1.f, true))
    lc.host_failure = true;
}

void heads_backward(LaunchCtx& lc, int prec, const NetDims& nd, const float* theta,
                    const bf16* theta16, const void* h, int n, const float* dz, const float* dV, void* gact_fc,
                    float* grad, float* scratch, GradSegments* segs) {
  if (prec == PAAC_BF16)
    heads_backward_t<bf16, bf16>(lc, nd, theta16, (const bf16*)h, n, dz, dV, (bf16*)gact_fc, grad, scratch, segs);
  else
    heads_backward_t<float, float>(lc, nd, theta, (const float*)h, n, dz, dV, (float*)gact_fc, grad, scratch, segs);
}

}  // namespace paac
