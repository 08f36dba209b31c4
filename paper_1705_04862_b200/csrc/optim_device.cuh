// What the kernels that close an update share: the clipping factor from the partial sums of the squared gradient, and the
// RMSProp step of one parameter.
#pragma once
#include "common.cuh"

namespace paac {

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
// The error word is the one the finishing kernel took down, not the live one: a block of the closing kernel itself may
// raise the range bit while others are still to read it.
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

}  // namespace paac
