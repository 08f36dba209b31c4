// Global-norm clipping + RMSProp for callers that must not allocate device memory.
//
// Some users of this library run where cudaMalloc is off limits: inside a real-time control loop that
// was promised a fixed memory footprint, inside a host process whose memory pool is owned by another
// framework and fully handed out, or in a sandbox that only lets pre-built modules touch the device.
// They cannot give the optimiser its scratch (the per-block partial sums of the squared gradient).  This
// file therefore carries that scratch itself, as a file-scope __device__ array that is part of the loaded
// module: every GPU that loads the library holds these 16 KB until the process exits, and no call here
// allocates or frees anything, on the device or through a library.
#include "common.cuh"
#include "per_device.h"

namespace {

constexpr int NA_SLICE = 4096;                        // parameters per partial sum at full capacity
constexpr int NA_MAX_SLICES = 4096;                   // capacity of the static scratch
constexpr size_t NA_MAX_PARAMS = (size_t)NA_SLICE * NA_MAX_SLICES;   // 16,777,216
constexpr int NA_THREADS = 256;

// One partial sum per block of the first launch.  Shared by every call on the device and never cleared: each call overwrites
// the entries it will read before reading them, so stale contents are harmless, but two calls that overlap
// on the GPU (different streams) would overwrite each other's sums.
static __device__ __align__(256) float g_noalloc_partials[NA_MAX_SLICES];

// In host code the array's name is only a handle for the runtime; the device address has to be asked for,
// once per device, with that device current.
paac::PerDevice<float*> g_partials_addr;

int partials_for_current_device(float** out) {
  int dev = -1;
  float* const* p = nullptr;
  if (cudaGetDevice(&dev) == cudaSuccess)
    p = g_partials_addr.get(dev, [](float*& at) {
      void* found = nullptr;
      if (cudaGetSymbolAddress(&found, g_noalloc_partials) != cudaSuccess) return false;
      at = static_cast<float*>(found);
      return at != nullptr;
    });
  if (p == nullptr) { cudaGetLastError(); return PAAC_ERR_CUDA; }
  *out = *p;
  return PAAC_OK;
}

// Two launches.  The first adds up the squares; the second is launched so that it may start while the first runs: its
// threads fetch their parameters, state and gradients, which the first does not write, and only then wait for the sum.
// What is left after the wait is arithmetic and stores.  What bounds it: two launches of latency (about 5 us) up to some
// hundred thousand parameters, then memory: 20 bytes read and written per parameter, the gradient a second time from L2.
// 1.69 M parameters with the bf16 copy: 17.5 us with 4-byte accesses and the second launch waiting for the first to
// end, 10.2 us with that, 8.8 us now that the first launch is made early too (4 M: 22.5 and 21.0 us, 20,000: 7.6 and 7.0).
// Arrays that are not all 16-byte aligned (8 for the bf16 copy) take the same kernels one element at a time.
constexpr int NA_SUM_BLOCKS = 592, NA_UPD_THREADS = 512, NA_UPD_BLOCKS = 296, NA_AHEAD = 3;
static_assert(NA_SUM_BLOCKS <= NA_MAX_SLICES, "the partial sums fit");

template <int W> struct Vec;
template <> struct Vec<4> { typedef float4 F; typedef uint2 H; };
template <> struct Vec<1> { typedef float F; typedef uint16_t H; };

__device__ __forceinline__ float block_sum(float acc, float* sh /* [32] */) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
  __syncthreads();
  float t = 0.f;
  for (unsigned w = 0; w < blockDim.x / 32; ++w) t += sh[w];        // the same order in every thread
  return t;
}
template <int W> __device__ __forceinline__ float sum_squares(const float* g, size_t n, size_t first, size_t stride) {
  typedef typename Vec<W>::F V;
  float acc = 0.f;
  const size_t nv = n / W;
#pragma unroll 4
  for (size_t i = first; i < nv; i += stride) {
    const V v = reinterpret_cast<const V*>(g)[i];
    const float* x = reinterpret_cast<const float*>(&v);
#pragma unroll
    for (int j = 0; j < W; ++j) acc = fmaf(x[j], x[j], acc);
  }
  for (size_t i = nv * W + first; i < n; i += stride) acc = fmaf(g[i], g[i], acc);
  return acc;
}
// m <- rho m + (1 - rho)(scale g)^2, theta <- theta - lr (scale g) / sqrt(m + eps)
struct NaStep {
  float lr, rho, eps, scale;
  __device__ __forceinline__ void operator()(float& t, float& m, float g) const {
    const float gs = scale * g;
    m = fmaf(rho, m, (1.f - rho) * gs * gs);
    t = t - lr * gs / sqrtf(m + eps);
  }
};
__device__ __forceinline__ float na_scale(float total, float clip, float* norm_and_scale) {
  const float norm = sqrtf(total);
  const bool ok = isfinite(norm);
  float scale = 1.f;
  if (ok && clip > 0.f && norm > clip) scale = clip / norm;
  if (blockIdx.x == 0 && threadIdx.x == 0 && norm_and_scale != nullptr) { norm_and_scale[0] = norm; norm_and_scale[1] = ok ? scale : 0.f; }
  return ok ? scale : -1.f;                          // non-finite norm: leave everything as it is
}
template <int W> __device__ __forceinline__ void store_half(uint16_t* half, size_t i, const float* t) {
  uint16_t h[W];
#pragma unroll
  for (int j = 0; j < W; ++j) h[j] = __bfloat16_as_ushort(__float2bfloat16_rn(t[j]));
  if constexpr (W == 4) reinterpret_cast<uint2*>(half)[i] = make_uint2(h[0] | ((uint32_t)h[1] << 16), h[2] | ((uint32_t)h[3] << 16));
  else half[i] = h[0];
}

template <int W>
__global__ void __launch_bounds__(NA_THREADS)
noalloc_sumsq_kernel(const float* g, size_t n, float* partials) {
  paac::pdl_entry();
  __shared__ float sh[32];
  const float t = block_sum(sum_squares<W>(g, n, blockIdx.x * (size_t)NA_THREADS + threadIdx.x, (size_t)gridDim.x * NA_THREADS), sh);
  if (threadIdx.x == 0) partials[blockIdx.x] = t;
}

template <int W>
__global__ void __launch_bounds__(NA_UPD_THREADS, 2)
noalloc_update_kernel(float* theta, float* rms, const float* g, uint16_t* theta_bf16, size_t n, float lr, float rho, float eps,
                      float clip, const float* partials, int n_partials, float* norm_and_scale) {
  typedef typename Vec<W>::F V;
  __shared__ float sh[32];
  const size_t nv = n / W, i0 = blockIdx.x * (size_t)NA_UPD_THREADS + threadIdx.x, stride = (size_t)gridDim.x * NA_UPD_THREADS;
  V gv[NA_AHEAD], mv[NA_AHEAD], tv[NA_AHEAD];
#pragma unroll
  for (int u = 0; u < NA_AHEAD; ++u) {
    const size_t i = i0 + u * stride;
    if (i < nv) { gv[u] = reinterpret_cast<const V*>(g)[i]; mv[u] = reinterpret_cast<V*>(rms)[i]; tv[u] = reinterpret_cast<V*>(theta)[i]; }
  }
  paac::pdl_entry();
  float acc = 0.f;
  for (int i = threadIdx.x; i < n_partials; i += NA_UPD_THREADS) acc += partials[i];
  const NaStep step{lr, rho, eps, na_scale(block_sum(acc, sh), clip, norm_and_scale)};
  if (step.scale < 0.f) return;
  auto apply = [&](size_t i, V& t, V& m, const V& gr) {
    float* tp = reinterpret_cast<float*>(&t); float* mp = reinterpret_cast<float*>(&m); const float* gp = reinterpret_cast<const float*>(&gr);
#pragma unroll
    for (int j = 0; j < W; ++j) step(tp[j], mp[j], gp[j]);
    reinterpret_cast<V*>(rms)[i] = m; reinterpret_cast<V*>(theta)[i] = t;
    if (theta_bf16 != nullptr) store_half<W>(theta_bf16, i, tp);
  };
#pragma unroll
  for (int u = 0; u < NA_AHEAD; ++u)
    if (i0 + u * stride < nv) apply(i0 + u * stride, tv[u], mv[u], gv[u]);
  for (size_t i = i0 + NA_AHEAD * stride; i < nv; i += stride) {
    V t = reinterpret_cast<V*>(theta)[i], m = reinterpret_cast<V*>(rms)[i];
    apply(i, t, m, reinterpret_cast<const V*>(g)[i]);
  }
  if (W > 1 && i0 < n - nv * W) {
    const size_t i = nv * W + i0;
    float t = theta[i], m = rms[i];
    step(t, m, g[i]);
    rms[i] = m; theta[i] = t;
    if (theta_bf16 != nullptr) theta_bf16[i] = __bfloat16_as_ushort(__float2bfloat16_rn(t));
  }
}

// Up to NA_ONE_BLOCK parameters one block does it all in one launch, its elements kept in registers between the two
// passes: below that size a second launch costs more than the rest of the device would save.
constexpr int NA_ONE_BLOCK = 8192, NA_ONE_THREADS = 1024;
__global__ void __launch_bounds__(NA_ONE_THREADS)
noalloc_one_block_kernel(float* theta, float* rms, const float* g, uint16_t* theta_bf16, int n, float lr, float rho, float eps,
                         float clip, float* norm_and_scale) {
  constexpr int PER = NA_ONE_BLOCK / NA_ONE_THREADS;
  __shared__ float sh[32];
  paac::pdl_entry();
  float gv[PER], mv[PER], tv[PER], acc = 0.f;
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int i = threadIdx.x + u * NA_ONE_THREADS;
    gv[u] = mv[u] = tv[u] = 0.f;
    if (i < n) { gv[u] = g[i]; mv[u] = rms[i]; tv[u] = theta[i]; }
  }
#pragma unroll
  for (int u = 0; u < PER; ++u) acc = fmaf(gv[u], gv[u], acc);
  const NaStep step{lr, rho, eps, na_scale(block_sum(acc, sh), clip, norm_and_scale)};
  if (step.scale < 0.f) return;
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int i = threadIdx.x + u * NA_ONE_THREADS;
    if (i < n) {
      step(tv[u], mv[u], gv[u]);
      rms[i] = mv[u]; theta[i] = tv[u];
      if (theta_bf16 != nullptr) theta_bf16[i] = __bfloat16_as_ushort(__float2bfloat16_rn(tv[u]));
    }
  }
}

template <int W>
cudaError_t two_launches(float* theta, float* rms, const float* grad, uint16_t* theta_bf16, size_t n, float lr, float rho, float eps,
                         float clip, float* partials, float* norm_and_scale, cudaStream_t s) {
  const size_t sums = (n / W + NA_THREADS - 1) / NA_THREADS, upds = (n / W + NA_UPD_THREADS - 1) / NA_UPD_THREADS;
  const int blocks = sums < NA_SUM_BLOCKS ? (int)sums : NA_SUM_BLOCKS;
  const cudaError_t summed = paac::launch_overlapped_on(s, noalloc_sumsq_kernel<W>, dim3(blocks), dim3(NA_THREADS), 0, grad, n, partials);
  if (summed != cudaSuccess) return summed;
  return paac::launch_overlapped_on(s, noalloc_update_kernel<W>, dim3(upds < NA_UPD_BLOCKS ? (unsigned)upds : NA_UPD_BLOCKS), dim3(NA_UPD_THREADS), 0,
                                    theta, rms, grad, theta_bf16, n, lr, rho, eps, clip, partials, blocks, norm_and_scale);
}

}  // namespace

extern "C" int paac_clip_rmsprop_noalloc(float* theta, float* rms, const float* grad, uint16_t* theta_bf16, size_t n,
                                         float lr, float rms_decay, float rms_eps, float clip_norm,
                                         float* norm_and_scale, void* stream) {
  if (!theta || !rms || !grad || n == 0) return PAAC_ERR_ARG;
  if (n > NA_MAX_PARAMS) return PAAC_ERR_LIMIT;
  float* partials = nullptr;
  const int st = partials_for_current_device(&partials);
  if (st != PAAC_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const bool wide = (((uintptr_t)theta | (uintptr_t)rms | (uintptr_t)grad) & 15u) == 0 && ((uintptr_t)theta_bf16 & 7u) == 0;
  cudaError_t launched;
  if (n <= (size_t)NA_ONE_BLOCK)
    launched = paac::launch_overlapped_on(s, noalloc_one_block_kernel, dim3(1), dim3(NA_ONE_THREADS), 0, theta, rms, grad, theta_bf16, (int)n, lr, rms_decay,
                                          rms_eps, clip_norm, norm_and_scale);
  else if (wide)
    launched = two_launches<4>(theta, rms, grad, theta_bf16, n, lr, rms_decay, rms_eps, clip_norm, partials, norm_and_scale, s);
  else
    launched = two_launches<1>(theta, rms, grad, theta_bf16, n, lr, rms_decay, rms_eps, clip_norm, partials, norm_and_scale, s);
  return paac::launch_status(launched);
}

extern "C" size_t paac_noalloc_max_params(void) { return NA_MAX_PARAMS; }
