// Parameter initialisation and the synthetic hashed environment.
#include "env_device.cuh"
#include "kernels.h"

namespace paac {

// Xavier-uniform: element i of weight tensor `layer` is (2u-1)*bound with u the 24-bit
// Philox uniform of counter (i, layer, 0, RNG_STREAM_INIT).  2u-1 is exact in float, so the
// single rounding of the product is the same on any IEEE machine.
__global__ void xavier_kernel(float* w, uint32_t count, float bound, uint32_t layer, uint64_t seed) {
  pdl_entry();
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
    const float u = philox_uniform(i, layer, 0u, RNG_STREAM_INIT, seed);
    w[i] = __fmul_rn(__fsub_rn(__fmul_rn(2.0f, u), 1.0f), bound);
  }
}

static void xavier(LaunchCtx& lc, float* w, size_t count, double fan_in, double fan_out,
                   uint32_t layer, uint64_t seed) {
  const float bound = (float)sqrt(6.0 / (fan_in + fan_out));
  int blocks = (int)((count + 255) / 256);
  if (blocks > 1184) blocks = 1184;
  KernelScope scope(lc, KID_INIT);
  launch_kernel(lc, xavier_kernel, blocks, 256, 0, w, (uint32_t)count, bound, layer, seed);
}

void launch_init_params(LaunchCtx& lc, const NetDims& nd, uint64_t seed, float* theta) {
  cudaMemsetAsync(theta, 0, nd.P * sizeof(float), lc.st);
  uint32_t id = 0;
  for (int l = 0; l < nd.n_conv; ++l, ++id) {
    const LayerDims& d = nd.layer[l];
    const double kk = (double)d.K * d.K;
    xavier(lc, theta + d.w_off, (size_t)d.CO * d.K * d.K * d.C, kk * d.C, kk * d.CO, id, seed);
  }
  const LayerDims& f = nd.layer[nd.n_conv];
  const size_t in = (size_t)f.H * f.W * f.C;
  xavier(lc, theta + f.w_off, in * nd.F, (double)in, (double)nd.F, id++, seed);
  xavier(lc, theta + nd.pi_w, (size_t)nd.A * nd.F, (double)nd.F, (double)nd.A, id++, seed);
  xavier(lc, theta + nd.v_w, (size_t)nd.F, (double)nd.F, 1.0, id++, seed);
}

__global__ void cast_bf16_kernel(const float* src, bf16* dst, size_t n) {
  pdl_entry();
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    dst[i] = __float2bfloat16_rn(src[i]);
}
void launch_cast_bf16(LaunchCtx& lc, const float* src, bf16* dst, size_t n) {
  int blocks = (int)((n + 255) / 256);
  if (blocks > 1184) blocks = 1184;
  KernelScope scope(lc, KID_CAST);
  launch_kernel(lc, cast_bf16_kernel, blocks, 256, 0, src, dst, n);
}

// One block per environment.  The block's first thread decides reward and terminal flag of
// the transition (seed, env, step, action) and keeps the episode counters; all threads then
// write the 84x84x4 frame of the state reached, one hashed 32-bit word per pixel (its bytes,
// little endian, are the four channels), as 16-byte stores.
constexpr int ENV_THREADS = 256;

// With PARTS > 0 (SAMPLE) the block's first warp also takes the action first: it finishes the heads of its environment from the
// partial dot products hp[part][e][k] the fully connected kernel left (k < A policy rows, k = A value row;
// rows 32 floats apart), softmax, inverse-CDF draw from the Philox uniform of (env, step) exactly as the stand-alone
// sampling kernel does, and writes logits, value, uniform and action; the transition then uses that action.
template <int PARTS>
__global__ void __launch_bounds__(ENV_THREADS)
env_step_kernel(uint64_t seed, int n_e, const uint64_t* __restrict__ step_base, uint32_t t,
                const int32_t* actions, uint32_t term_denom,
                uint8_t* __restrict__ next_frames, int8_t* __restrict__ rewards, uint8_t* __restrict__ terminals,
                int32_t* __restrict__ counters, HeadsTail ht, int pattern_actions) {
  // Two roles run side by side until the action is known: the first warp takes it (SAMPLE), and the first thread of
  // the second warp prepares everything of the transition that does not depend on it -- the hash chains of this step
  // and the next up to the point where the action enters, and the environment's counters, whose loads would otherwise
  // be waited for after the draw.  One hash step, the reward / terminal bits and the frame's base remain.
  constexpr bool SAMPLE = PARTS > 0;
  __shared__ EnvFrame s_frame;
  __shared__ int32_t s_action;
  const uint32_t e = blockIdx.x;
  const bool stepping = SAMPLE || actions != nullptr;          // else: the start frames (step 0, tag 0)
  EnvPrep prep{};
  // what precedes the wait was written at least five kernels ago (the counters, the step index, the biases)
  if (SAMPLE && threadIdx.x == 32) prep = env_prepare(seed, e, n_e, (uint32_t)(*step_base) + t, counters);     // step index of this transition
  if (SAMPLE && threadIdx.x < 32) {
    const int lane = threadIdx.x, A = ht.A;
    const float bias = lane < A ? __ldg(ht.bpi + lane) : (lane == A ? __ldg(ht.bv) : 0.f);   // older than the previous kernel
    pdl_entry();
    float sum = -INFINITY;
    if (lane <= A) sum = sum_head_parts<SAMPLE ? PARTS : 2>(ht.hp, n_e, e, lane) + bias;
    const float z = lane < A ? sum : -INFINITY;
    const int32_t a = warp_finish_heads(ht.mode, z, __shfl_sync(0xffffffffu, sum, A), lane, A, (size_t)e, ht.logits, ht.values, true,
                                        seed, *step_base + t, ht.forced, ht.actions, ht.sampled, ht.uniforms);
    if (lane == 0) s_action = a;
  } else {
    pdl_entry();
    if (!SAMPLE && threadIdx.x == 32) {
      if (stepping) {
        prep = env_prepare(seed, e, n_e, (uint32_t)(*step_base) + t, counters);
        s_action = actions[e];
      } else {
        prep.pre_next = env_hash_prefix(seed, e, 0u);
      }
    }
  }
  __syncthreads();
  EnvOutcome o{0, false, 0u};
  if (threadIdx.x == 32) {
    if (stepping) o = env_outcome(prep, s_action, term_denom, pattern_actions);
    s_frame = env_frame_of(prep.pre_next, o.tag, pattern_actions);
  }
  __syncthreads();
  if (threadIdx.x == 32 && stepping) env_record(prep, o, e, n_e, rewards, terminals, counters);
  env_write_frame<ENV_THREADS>(s_frame, next_frames + (size_t)e * FRAME_BYTES, pattern_actions);
}

void launch_env_step(LaunchCtx& lc, uint64_t seed, int n_e, const uint64_t* step_base, uint32_t t,
                     const int32_t* actions, uint32_t term_denom, uint8_t* next_frames, int8_t* rewards,
                     uint8_t* terminals, int32_t* counters, int pattern_actions) {
  KernelScope scope(lc, KID_ENV_STEP);
  launch_kernel(lc, env_step_kernel<0>, n_e, ENV_THREADS, 0, seed, n_e, step_base, t, actions, term_denom, next_frames, rewards,
                                                  terminals, counters, HeadsTail{}, pattern_actions);
}

void launch_env_step_sampling(LaunchCtx& lc, uint64_t seed, int n_e, const uint64_t* step_base, uint32_t t, uint32_t term_denom,
                              uint8_t* next_frames, int8_t* rewards, uint8_t* terminals, int32_t* counters,
                              const HeadsTail& ht, int pattern_actions) {
  KernelScope scope(lc, KID_ENV_STEP);
  // up to two blocks per SM may set up while the previous kernel drains; more of them would pile up on the first free SMs
  auto kern = ht.parts == 2 ? env_step_kernel<2> : (ht.parts == 4 ? env_step_kernel<4> : env_step_kernel<8>);
  auto launch = [&](auto how) {
    how(lc, kern, dim3(n_e), dim3(ENV_THREADS), (size_t)0, seed, n_e, step_base, t, (const int32_t*)nullptr, term_denom, next_frames, rewards,
        terminals, counters, ht, pattern_actions);
  };
  if (n_e <= 296) launch([](auto&&... a) { launch_kernel_overlapped(a...); });
  else launch([](auto&&... a) { launch_kernel(a...); });
}

// the environments' global step index lives on the device, so that a recorded sequence of launches can be
// replayed for the next iteration without new arguments
__global__ void advance_step_kernel(uint64_t* step_base, uint32_t by) {
  pdl_entry(); *step_base += by; }
void launch_advance_step(LaunchCtx& lc, uint64_t* step_base, uint32_t by) {
  KernelScope scope(lc, KID_ENV_STEP);
  launch_kernel(lc, advance_step_kernel, 1, 1, 0, step_base, by);
}

}  // namespace paac
