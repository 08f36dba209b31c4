// Global-norm clipping fused with RMSProp.
#include <cuda_fp16.h>

#include "kernels.h"

namespace paac {

// Where four neighbouring parameters from element p on (outside the fully connected matrix) go in the regrouped images, as bf16 bits
__device__ __forceinline__ void small_images(const WeightImages& img, size_t p, const uint16_t (&b)[4]) {
  if (p < img.w1_end) {
    // [co][8][8][4]: a pixel's four channels, next to each other in w1_b[co][tap][py][px][ci] too, as fp16 times 2^8
    const int i = (int)p, sx = (i >> 2) & 7, r = (i >> 5) & 7, co = i >> 8;
    uint16_t h[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float scaled = __uint_as_float((uint32_t)b[j] << 16) * img.w1_scale;
      if (!(fabsf(scaled) <= 65504.f)) atomicOr(img.error_word, DEV_ERR_RANGE);      // beyond fp16 (or not a number)
      h[j] = __half_as_ushort(__float2half_rn(scaled));
    }
    uint16_t* to = img.w1_b + ((((co * 4 + 2 * (r >> 2) + (sx >> 2)) * 4 + (r & 3)) * 4 + (sx & 3)) << 2);
    *reinterpret_cast<uint2*>(to) = make_uint2(h[0] | ((uint32_t)h[1] << 16), h[2] | ((uint32_t)h[3] << 16));
  } else if (p >= img.w2_off && p < img.w2_off + NatConv2::KK * NatConv2::CO) {
    // W2[co][r][s][ci] -> w2_d[2 (r & 1) + (s & 1)][ci][2 (r >> 1) + (s >> 1)][co]
    const int i = (int)(p - img.w2_off), ci = i % 32, s = (i / 32) % 4, r = (i / 128) % 4, co = i / 512;
    uint16_t* to = img.w2_d + (((2 * (r & 1) + (s & 1)) * 32 + ci) * 4 + 2 * (r >> 1) + (s >> 1)) * 64 + co;
#pragma unroll
    for (int j = 0; j < 4; ++j) to[j * 256] = b[j];
  } else if (p >= img.w3_off && p < img.w3_off + NatConv3::KK * NatConv3::CO) {
    // W3[co][tap][ci] -> w3_d[ci][tap][co]
    const int i = (int)(p - img.w3_off), ci = i % 64, tap = (i / 64) % 9, co = i / 576;
    uint16_t* to = img.w3_d + (ci * 9 + tap) * 64 + co;
#pragma unroll
    for (int j = 0; j < 4; ++j) to[j * 576] = b[j];
  }
}

struct RmsStep {
  float lr, rho, eps, scale;
  // m <- rho m + (1 - rho) (scale g)^2,  theta <- theta - lr (scale g) / sqrt(m + eps)
  __device__ __forceinline__ void operator()(float& t, float& m, float g) const {
    const float gs = scale * g;
    m = fmaf(rho, m, (1.f - rho) * gs * gs);
    t = t - lr * gs / sqrtf(m + eps);
  }
};

// Every block re-adds the partials in the same order (so all agree bit for bit) and forms scale = min(1, clip / norm); -1
// means that parameters and state stay as they are: a non-finite norm, or a device error left by any earlier kernel (a
// bounded wait that gave up means some tile or partial sum of this update is garbage), which the status then names.
template <int THREADS>
__device__ __forceinline__ float clip_scale_of(const float* partials, int n_partials, float clip, uint32_t dev_err, DeviceStats* stats) {
  __shared__ float sh[THREADS / 32];
  __shared__ float s_scale;
  float acc = 0.f;
  for (int i = threadIdx.x; i < n_partials; i += THREADS) acc += partials[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    float total = 0.f;
#pragma unroll
    for (int w = 0; w < THREADS / 32; ++w) total += sh[w];
    const float norm = sqrtf(total);
    float scale = 1.f;
    const bool ok = isfinite(norm) && dev_err == 0u;
    if (ok && clip > 0.f && norm > clip) scale = clip / norm;
    s_scale = ok ? scale : -1.f;
    if (blockIdx.x == 0) {
      stats->grad_norm = norm;
      stats->clip_scale = ok ? scale : 0.f;
      stats->status = ok ? PAAC_OK
                         : ((dev_err & DEV_ERR_WAIT_MASK) ? PAAC_ERR_TIMEOUT
                                                           : ((dev_err & DEV_ERR_RANGE) ? PAAC_ERR_RANGE : PAAC_ERR_NONFINITE));
    }
  }
  __syncthreads();
  return s_scale;
}

// pass 2: norm, clipping factor, RMSProp and the refreshed bf16 copy.
// One wave of two blocks per SM, launched so that it may start while the finishing kernel drains: a thread's first
// UPD_AHEAD groups of parameters and state (all of them, up to 1.8 M parameters) are fetched before the wait, the
// gradients right after it, together with the partial sums of the norm.
constexpr int UPD_THREADS = 512, UPD_BLOCKS = 296, UPD_AHEAD = 3;
__global__ void __launch_bounds__(UPD_THREADS, 2)
clip_rmsprop_kernel(size_t P, float* theta, float* rms, const float* g,
                    bf16* __restrict__ theta16, float lr, float rho, float eps, float clip,
                    const float* partials, int n_partials, DeviceStats* stats) {
  const size_t n4 = P / 4, stride = (size_t)gridDim.x * UPD_THREADS;
  float4* t4 = reinterpret_cast<float4*>(theta);
  float4* m4 = reinterpret_cast<float4*>(rms);
  const float4* g4 = reinterpret_cast<const float4*>(g);
  const size_t i0 = blockIdx.x * (size_t)UPD_THREADS + threadIdx.x;
  float4 gv0[UPD_AHEAD], mv0[UPD_AHEAD], tv0[UPD_AHEAD];
#pragma unroll
  for (int u = 0; u < UPD_AHEAD; ++u)
    if (i0 + u * stride < n4) { mv0[u] = m4[i0 + u * stride]; tv0[u] = t4[i0 + u * stride]; }
  pdl_entry();
#pragma unroll
  for (int u = 0; u < UPD_AHEAD; ++u)
    if (i0 + u * stride < n4) gv0[u] = g4[i0 + u * stride];
  const RmsStep step{lr, rho, eps, clip_scale_of<UPD_THREADS>(partials, n_partials, clip, stats->error_word, stats)};
  if (step.scale < 0.f) return;
  auto apply = [&](size_t i, float4& tv, float4& mv, const float4& gv) {
    const float* gp = &gv.x; float* mp = &mv.x; float* tp = &tv.x;
#pragma unroll
    for (int j = 0; j < 4; ++j) step(tp[j], mp[j], gp[j]);
    m4[i] = mv; t4[i] = tv;
    if (theta16 != nullptr) {
      __nv_bfloat162 lo = __floats2bfloat162_rn(tv.x, tv.y), hi = __floats2bfloat162_rn(tv.z, tv.w);
      uint2 pk;
      pk.x = *reinterpret_cast<uint32_t*>(&lo); pk.y = *reinterpret_cast<uint32_t*>(&hi);
      reinterpret_cast<uint2*>(theta16)[i] = pk;
    }
  };
#pragma unroll
  for (int u = 0; u < UPD_AHEAD; ++u)
    if (i0 + u * stride < n4) apply(i0 + u * stride, tv0[u], mv0[u], gv0[u]);
  for (size_t i = i0 + UPD_AHEAD * stride; i < n4; i += stride) {
    float4 tv = t4[i], mv = m4[i];
    apply(i, tv, mv, g4[i]);
  }
  if (blockIdx.x == 0) {
    for (size_t i = n4 * 4 + threadIdx.x; i < P; i += UPD_THREADS) {
      float t = theta[i], m = rms[i];
      step(t, m, g[i]);
      rms[i] = m; theta[i] = t;
      if (theta16 != nullptr) theta16[i] = __float2bfloat16_rn(t);
    }
  }
}

// The same for the larger network's bf16 copies: the regrouped weight images (relayout_weights_kernel in net_tc.cu says which) are
// written from the new parameters as they are made, where a kernel of its own read the copies back, 5.7 us behind this one (an
// iteration of one learner: 32 environments 154.8 -> 151.3 us; at 256 and 1024 no more than runs differ by).  The fully
// connected matrix goes in tiles of 32 units x 64 inputs, a thread's float4 in each of up to three of them, so that its
// transpose leaves through shared memory in runs of 64 bytes; the blocks that have only two tiles take the rest of the
// parameters, whose images are small enough for scattered stores.  Arithmetic per parameter is that of clip_rmsprop_kernel.
constexpr int IMG_IN = 3136, IMG_OUT = 512, IMG_TI = 64, IMG_TO = 32, IMG_TILES = (IMG_IN / IMG_TI) * (IMG_OUT / IMG_TO), IMG_PITCH = IMG_TO + 2;
constexpr int IMG_FULL = IMG_TILES - (UPD_AHEAD - 1) * UPD_BLOCKS;       // blocks with a third tile
static_assert(IMG_IN % IMG_TI == 0 && IMG_TO * IMG_TI / 4 == UPD_THREADS && IMG_FULL > 0 && IMG_FULL < UPD_BLOCKS, "tiles and blocks");
__global__ void __launch_bounds__(UPD_THREADS, 2)
clip_rmsprop_images_kernel(size_t P, float* theta, float* rms, const float* g, bf16* __restrict__ theta16, WeightImages img, float lr, float rho,
                           float eps, float clip, const float* partials, int n_partials, DeviceStats* stats) {
  __shared__ uint16_t turned[UPD_AHEAD][IMG_TI][IMG_PITCH];
  const int tid = threadIdx.x;
  const size_t n4 = P / 4, fc4 = img.fc_off / 4, fc_end4 = fc4 + (size_t)IMG_IN * IMG_OUT / 4;
  float4* t4 = reinterpret_cast<float4*>(theta);
  float4* m4 = reinterpret_cast<float4*>(rms);
  const float4* g4 = reinterpret_cast<const float4*>(g);
  size_t at[UPD_AHEAD];
#pragma unroll
  for (int u = 0; u < UPD_AHEAD; ++u) {
    const int tile = blockIdx.x + u * UPD_BLOCKS;
    if (tile < IMG_TILES) {
      at[u] = fc4 + ((size_t)(tile % (IMG_OUT / IMG_TO)) * IMG_TO + tid / (IMG_TI / 4)) * (IMG_IN / 4) + tile / (IMG_OUT / IMG_TO) * (IMG_TI / 4) + tid % (IMG_TI / 4);
    } else {
      const size_t j = (size_t)(tile - IMG_TILES) * UPD_THREADS + tid;   // before the matrix, then behind it
      at[u] = j < fc4 ? j : fc_end4 + (j - fc4);
    }
  }
  float4 gv[UPD_AHEAD], mv[UPD_AHEAD], tv[UPD_AHEAD];
#pragma unroll
  for (int u = 0; u < UPD_AHEAD; ++u)
    if (at[u] < n4) { mv[u] = m4[at[u]]; tv[u] = t4[at[u]]; }
  pdl_entry();
#pragma unroll
  for (int u = 0; u < UPD_AHEAD; ++u)
    if (at[u] < n4) gv[u] = g4[at[u]];
  const RmsStep step{lr, rho, eps, clip_scale_of<UPD_THREADS>(partials, n_partials, clip, stats->error_word, stats)};
  if (step.scale < 0.f) return;
#pragma unroll
  for (int u = 0; u < UPD_AHEAD; ++u) {
    if (at[u] >= n4) continue;
    const float* gp = &gv[u].x; float* mp = &mv[u].x; float* tp = &tv[u].x;
    uint16_t b[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) { step(tp[j], mp[j], gp[j]); b[j] = __bfloat16_as_ushort(__float2bfloat16_rn(tp[j])); }
    m4[at[u]] = mv[u]; t4[at[u]] = tv[u];
    reinterpret_cast<uint2*>(theta16)[at[u]] = make_uint2(b[0] | ((uint32_t)b[1] << 16), b[2] | ((uint32_t)b[3] << 16));
    if (blockIdx.x + u * UPD_BLOCKS < IMG_TILES) {
#pragma unroll
      for (int j = 0; j < 4; ++j) turned[u][4 * (tid % (IMG_TI / 4)) + j][tid / (IMG_TI / 4)] = b[j];
    } else {
      small_images(img, at[u] * 4, b);
    }
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < UPD_AHEAD; ++u) {
    const int tile = blockIdx.x + u * UPD_BLOCKS, r = tid / 8, c = tid % 8;
    if (tile >= IMG_TILES) break;
    const uint32_t* from = reinterpret_cast<const uint32_t*>(&turned[u][r][4 * c]);
    *reinterpret_cast<uint2*>(img.wfc_t + (size_t)(tile / (IMG_OUT / IMG_TO) * IMG_TI + r) * IMG_OUT + tile % (IMG_OUT / IMG_TO) * IMG_TO + 4 * c) = make_uint2(from[0], from[1]);
  }
  if (blockIdx.x == 0)
    for (size_t i = n4 * 4 + tid; i < P; i += UPD_THREADS) {
      float t = theta[i], m = rms[i];
      step(t, m, g[i]);
      rms[i] = m; theta[i] = t;
      theta16[i] = __float2bfloat16_rn(t);
    }
}

void launch_clip_rmsprop_images(LaunchCtx& lc, size_t P, float* theta, float* rms, const float* grad, bf16* theta16, const WeightImages& img, float lr,
                                float rho, float eps, float clip, const float* norm_partials, DeviceStats* stats, int ready_partials) {
  KernelScope scope(lc, KID_CLIP_RMSPROP);
  launch_kernel_overlapped(lc, clip_rmsprop_images_kernel, UPD_BLOCKS, UPD_THREADS, 0, P, theta, rms, grad, theta16, img, lr, rho, eps, clip,
                           norm_partials, ready_partials, stats);
}

void launch_clip_rmsprop(LaunchCtx& lc, size_t P, float* theta, float* rms, const float* grad,
                         bf16* theta16, float lr, float rho, float eps, float clip, const float* norm_partials,
                         DeviceStats* stats, int ready_partials) {
  KernelScope scope(lc, KID_CLIP_RMSPROP);
  launch_kernel_overlapped(lc, clip_rmsprop_kernel, UPD_BLOCKS, UPD_THREADS, 0, P, theta, rms, grad, theta16, lr, rho, eps, clip,
                                                              norm_partials, ready_partials, stats);
}

}  // namespace paac
