// Frame pre-processing (Section 5.1 of the paper): per-pixel maximum of the two latest raw frames, pixel intensity,
// 210 x 160 -> 84 x 84, newest channel of the four-frame state.  Integer arithmetic throughout.
#include "env_device.cuh"
#include "kernels.h"
#include "per_device.h"

namespace paac {

constexpr int PP_SH = 210, PP_SW = 160, PP_BAND_OUT = 12, PP_BAND_SRC = 30, PP_BANDS = 7, PP_THREADS = 256;
constexpr int PP_RAW_BYTES = PP_SH * PP_SW * 3, PP_BAND_BYTES = PP_BAND_SRC * PP_SW * 3;       // 100,800 and 14,400
static_assert(PP_BANDS * PP_BAND_OUT == FRAME_H && PP_BANDS * PP_BAND_SRC == PP_SH, "bands tile the frame");
static_assert(PP_BAND_BYTES % 16 == 0 && PP_RAW_BYTES % 16 == 0, "16-byte loads");

// A task is one band of 12 output rows of one environment.  84 / 210 = 2 / 5, so a band reads exactly 30 source rows,
// one contiguous run of 14,400 bytes in each raw frame.  Rows: output row 2 m averages source rows 5 m, 5 m + 1, 5 m + 2
// with weights 2, 2, 1 and output row 2 m + 1 rows 5 m + 2 .. 5 m + 4 with weights 1, 2, 2.  Columns: in units of 1/21 of
// a source pixel, output column x covers [40 x, 40 x + 40) and source column c covers [21 c, 21 c + 21).  The weights add
// up to 5 x 40, and (sum + 100) / 200 is the area average rounded half up.
// What bounds it: memory, once enough of it is in flight.  Two resident blocks per SM walk the tasks; the raw bytes of
// the next PP_STAGES - 1 tasks are always on their way into shared memory (16-byte asynchronous copies) while a task goes
// through three passes: channel-wise maximum and intensity, sixteen pixels per thread (one dot-product instruction per
// pixel); the weighted sum over three rows, four columns per thread, two 16-bit sums per word; the weighted sum over at
// most three columns, one output pixel per thread.  One block per task with the loads at its front and nine byte reads
// per output pixel took 66 us for 1024 environments (264 MB); this takes 49.1 us in a row of calls on the same buffers, 46.6 with the
// set-up beside the end of the call before (51.0 where the buffers are others each time).
constexpr int PP_STAGES = 3, PP_ITEMS = PP_BAND_SRC * PP_SW / 16, PP_OUT = PP_BAND_OUT * FRAME_W;
constexpr int PP_OUT_PER = (PP_OUT + PP_THREADS - 1) / PP_THREADS;
struct PpShared {
  uint4 raw[PP_STAGES][2][PP_BAND_BYTES / 16];
  uint32_t grey[PP_BAND_SRC][PP_SW / 4];
  uint16_t rows[PP_BAND_OUT][PP_SW + 2];            // weighted sums over rows; the two columns past the end have weight 0
};
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
// channel-wise maximum of four bytes, as two pairs of 16-bit values
__device__ __forceinline__ uint32_t max_bytes(uint32_t a, uint32_t b) {
  const uint32_t even = __vmaxu2(a & 0x00FF00FFu, b & 0x00FF00FFu), odd = __vmaxu2((a >> 8) & 0x00FF00FFu, (b >> 8) & 0x00FF00FFu);
  return even | (odd << 8);
}

__global__ void __launch_bounds__(PP_THREADS, 2)
preprocess_kernel(const uint8_t* __restrict__ raw_prev, const uint8_t* __restrict__ raw_last,
                  const uint8_t* state_in, uint8_t* state_out, int tasks) {
  extern __shared__ __align__(16) unsigned char pp_smem[];
  PpShared& sm = *reinterpret_cast<PpShared*>(pp_smem);
  const int tid = threadIdx.x;
  auto request = [&](int task, int stage) {
    if (task < tasks) {
      const size_t src = (size_t)(task / PP_BANDS) * PP_RAW_BYTES + (size_t)(task % PP_BANDS) * PP_BAND_BYTES;
      for (int i = tid; i < PP_BAND_BYTES / 16; i += PP_THREADS) {
        cp_async16(&sm.raw[stage][0][i], raw_prev + src + 16 * (size_t)i);
        cp_async16(&sm.raw[stage][1][i], raw_last + src + 16 * (size_t)i);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (tid < PP_BAND_OUT * 2) sm.rows[tid >> 1][PP_SW + (tid & 1)] = 0;
  pdl_entry();
  for (int k = 0; k < PP_STAGES - 1; ++k) request(blockIdx.x + k * gridDim.x, k);
  int stage = 0;
  for (int task = blockIdx.x; task < tasks; task += gridDim.x, stage = stage + 1 == PP_STAGES ? 0 : stage + 1) {
    // the old state's words of this thread's output pixels, fetched while the passes before their use run
    const size_t pix0 = (size_t)(task / PP_BANDS) * FRAME_H * FRAME_W + (size_t)(task % PP_BANDS) * PP_OUT;
    uint32_t old[PP_OUT_PER];
    if (state_in != nullptr) {
#pragma unroll
      for (int u = 0; u < PP_OUT_PER; ++u)
        if (tid + u * PP_THREADS < PP_OUT) old[u] = reinterpret_cast<const uint32_t*>(state_in)[pix0 + tid + u * PP_THREADS];
    }
    asm volatile("cp.async.wait_group %0;" ::"n"(PP_STAGES - 2) : "memory");
    __syncthreads();                                 // the task's bytes are in; everyone is done with the stage before
    request(task + (PP_STAGES - 1) * gridDim.x, (stage + PP_STAGES - 1) % PP_STAGES);
    for (int i = tid; i < PP_ITEMS; i += PP_THREADS) {
      uint32_t w[13];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const uint4 a = sm.raw[stage][0][3 * i + k], b = sm.raw[stage][1][3 * i + k];
        w[4 * k] = max_bytes(a.x, b.x); w[4 * k + 1] = max_bytes(a.y, b.y);
        w[4 * k + 2] = max_bytes(a.z, b.z); w[4 * k + 3] = max_bytes(a.w, b.w);
      }
      w[12] = 0u;
      uint32_t g[4];
#pragma unroll
      for (int p4 = 0; p4 < 4; ++p4) {
        uint32_t y[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int byte = 3 * (4 * p4 + j), at = byte & 3;               // R, G, B and one byte more, which weighs 0
          const uint32_t rgb = at == 0 ? w[byte >> 2] : __funnelshift_r(w[byte >> 2], w[(byte >> 2) + 1], 8 * at);
          y[j] = __dp4a(rgb, 0x001D964Du, 128u);                          // 77 R + 150 G + 29 B + 128, below 2^16
        }
        g[p4] = __byte_perm(__byte_perm(y[0], y[1], 0x0051), __byte_perm(y[2], y[3], 0x0051), 0x5410);
      }
      reinterpret_cast<uint4*>(&sm.grey[0][0])[i] = make_uint4(g[0], g[1], g[2], g[3]);
    }
    __syncthreads();
    for (int i = tid; i < PP_BAND_OUT * PP_SW / 4; i += PP_THREADS) {
      const int yl = i / (PP_SW / 4), c4 = i % (PP_SW / 4), odd = yl & 1;
      const int r0 = 5 * (yl >> 1) + 2 * odd;                             // three source rows r0 .. r0 + 2
      const uint32_t a = sm.grey[r0][c4], b = sm.grey[r0 + 1][c4], c = sm.grey[r0 + 2][c4];
      const uint32_t wa = odd ? 1u : 2u, wc = odd ? 2u : 1u;              // the middle one always weighs 2
      const uint32_t even = (a & 0x00FF00FFu) * wa + (b & 0x00FF00FFu) * 2u + (c & 0x00FF00FFu) * wc;
      const uint32_t odds = ((a >> 8) & 0x00FF00FFu) * wa + ((b >> 8) & 0x00FF00FFu) * 2u + ((c >> 8) & 0x00FF00FFu) * wc;
      uint32_t* dst = reinterpret_cast<uint32_t*>(&sm.rows[yl][4 * c4]);
      dst[0] = __byte_perm(even, odds, 0x5410); dst[1] = __byte_perm(even, odds, 0x7632);
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < PP_OUT_PER; ++u) {
      const int o = tid + u * PP_THREADS;
      if (o >= PP_OUT) break;
      const int yl = o / FRAME_W, x = o - yl * FRAME_W;
      const int u0 = 40 * x, c0 = u0 / 21;                                // first source column; at most three are touched
      const uint32_t first = (uint32_t)(21 * c0 + 21 - u0);              // what of the box lies in it: 1 .. 21
      const uint32_t second = min(40u - first, 21u), third = 40u - first - second;
      const uint16_t* r = &sm.rows[yl][c0];
      const uint32_t v = (first * r[0] + second * r[1] + third * r[2] + 100u) / 200u;
      uint32_t out;
      if (state_in != nullptr) out = (old[u] >> 8) | (v << 24);           // channels are bytes, oldest first
      else out = v * 0x01010101u;
      reinterpret_cast<uint32_t*>(state_out)[pix0 + o] = out;
    }
  }
}

// The frame stack by itself: out = (the three newest channels of prev, newest), or four copies of newest where the
// environment restarts.  A thread takes four pixels: one 16-byte load of the previous state, one 4-byte load of the
// new plane, one 16-byte store.  prev == out is allowed (every word is read before it is written, by the same thread).
constexpr int SP_THREADS = 256, SP_QUADS = FRAME_H * FRAME_W / 4;          // 1764 groups of four pixels per state
__global__ void __launch_bounds__(SP_THREADS)
stack_push_kernel(const uint8_t* prev, const uint8_t* __restrict__ newest, const uint8_t* __restrict__ restart,
                  uint8_t* out) {
  pdl_entry();
  const uint32_t e = blockIdx.y;
  const bool fresh = restart != nullptr && restart[e] != 0;
  const uint4* src = reinterpret_cast<const uint4*>(prev + (size_t)e * FRAME_BYTES);
  const uint32_t* nw = reinterpret_cast<const uint32_t*>(newest + (size_t)e * FRAME_H * FRAME_W);
  uint4* dst = reinterpret_cast<uint4*>(out + (size_t)e * FRAME_BYTES);
  for (int q = blockIdx.x * SP_THREADS + threadIdx.x; q < SP_QUADS; q += gridDim.x * SP_THREADS) {
    const uint32_t v = nw[q];
    uint4 w;
    if (fresh) {
      w = make_uint4((v & 0xFFu) * 0x01010101u, ((v >> 8) & 0xFFu) * 0x01010101u, ((v >> 16) & 0xFFu) * 0x01010101u,
                     (v >> 24) * 0x01010101u);
    } else {
      const uint4 p = src[q];
      w = make_uint4((p.x >> 8) | (v << 24), (p.y >> 8) | ((v >> 8) << 24), (p.z >> 8) | ((v >> 16) << 24),
                     (p.w >> 8) | ((v >> 24) << 24));
    }
    dst[q] = w;
  }
}

// The same for the external-environment mode, sixteen pixels per thread and all of a thread's plane words asked for before
// any is used: they come over the host link, whose latency is a microsecond or two and whose bandwidth (about 50 GB/s) is
// what bounds the kernel from a few dozen environments on.  Which stacks start afresh comes as a launch argument, as does
// where the planes are: read by every block from pinned memory, they cost 130 ns a block (reads of one address are served
// one after the other) and as much for every warp's flags (1024 environments: 158 us, 147 without; 32: 10 us, 3 within rollout_tc_kernel).
constexpr int PULL_AHEAD = 3, PULL_BLOCKS = 592, PULL_ENVS = 2048;
struct PullFresh { uint32_t bits[PULL_ENVS / 32]; };
__global__ void __launch_bounds__(SP_THREADS)
stack_pull_kernel(const uint8_t* prev, const uint8_t* planes, const __grid_constant__ PullFresh fresh, uint8_t* out, int n) {
  pdl_entry();
  const uint32_t items = (uint32_t)n * STACK_ITEMS, stride = gridDim.x * SP_THREADS;
  const uint4* newest = reinterpret_cast<const uint4*>(planes);
  for (uint32_t base = blockIdx.x * SP_THREADS + threadIdx.x; base < items; base += PULL_AHEAD * stride) {
    uint4 v[PULL_AHEAD];
#pragma unroll
    for (int u = 0; u < PULL_AHEAD; ++u)
      if (base + u * stride < items) v[u] = newest[base + u * stride];
#pragma unroll
    for (int u = 0; u < PULL_AHEAD; ++u) {
      const uint32_t i = base + u * stride;
      if (i >= items) break;
      const uint32_t e = i / STACK_ITEMS;
      stack_sixteen(v[u], (fresh.bits[e >> 5] >> (e & 31u)) & 1u, reinterpret_cast<const uint4*>(prev) + (size_t)i * 4, reinterpret_cast<uint4*>(out) + (size_t)i * 4);
    }
  }
}
void launch_stack_pull(LaunchCtx& lc, const uint8_t* prev, const uint8_t* planes, const uint8_t* restart, uint8_t* out, int n) {
  for (int e0 = 0; e0 < n; e0 += PULL_ENVS) {
    const int count = n - e0 < PULL_ENVS ? n - e0 : PULL_ENVS;
    PullFresh fresh{};
    if (restart)
      for (int e = 0; e < count; ++e) fresh.bits[e >> 5] |= (uint32_t)(restart[e0 + e] != 0) << (e & 31);
    const size_t blocks = ((size_t)count * STACK_ITEMS + SP_THREADS - 1) / SP_THREADS, at = (size_t)e0 * FRAME_BYTES;
    KernelScope scope(lc, KID_ENV_STEP);
    launch_kernel(lc, stack_pull_kernel, dim3(blocks < PULL_BLOCKS ? (unsigned)blocks : PULL_BLOCKS), dim3(SP_THREADS), 0, prev + at,
                  planes + at / FRAME_C, fresh, out + at, count);
  }
}

// one block: a few kilobytes of posted writes over the host link, made visible before the flag
constexpr int PUB_THREADS = 512;
__global__ void __launch_bounds__(PUB_THREADS)
publish_kernel(const int32_t* actions, const float* values, int n, int32_t* host_actions, float* host_values, volatile uint32_t* done) {
  pdl_entry();
  for (int i = threadIdx.x; i < n; i += PUB_THREADS) {
    if (actions != nullptr) host_actions[i] = actions[i];
    host_values[i] = values[i];
  }
  __threadfence_system();
  __syncthreads();
  if (threadIdx.x == 0) *done = 1u;
}
void launch_publish(LaunchCtx& lc, const int32_t* actions, const float* values, int n, int32_t* host_actions, float* host_values,
                    volatile uint32_t* done) {
  KernelScope scope(lc, KID_HEADS_FWD);
  launch_kernel_overlapped(lc, publish_kernel, dim3(1), dim3(PUB_THREADS), 0, actions, values, n, host_actions, host_values, done);
}

__global__ void __launch_bounds__(32) publish_stats_kernel(const DeviceStats* stats, DeviceStats* host_stats, volatile uint32_t* done) {
  constexpr int WORDS = sizeof(DeviceStats) / 4;
  static_assert(WORDS <= 32, "one word per lane");
  pdl_entry();
  if (threadIdx.x < WORDS) reinterpret_cast<uint32_t*>(host_stats)[threadIdx.x] = reinterpret_cast<const uint32_t*>(stats)[threadIdx.x];
  __threadfence_system();
  __syncwarp();
  if (threadIdx.x == 0) *done = 1u;
}
void launch_publish_stats(LaunchCtx& lc, const DeviceStats* stats, DeviceStats* host_stats, volatile uint32_t* done) {
  KernelScope scope(lc, KID_CLIP_RMSPROP);
  launch_kernel_overlapped(lc, publish_stats_kernel, dim3(1), dim3(32), 0, stats, host_stats, done);
}

}  // namespace paac

extern "C" int paac_stack_push(const uint8_t* state_in, const uint8_t* newest, const uint8_t* restart, uint8_t* state_out,
                               int n, void* stream) {
  using namespace paac;
  if (!state_in || !newest || !state_out || n < 1 || n > 65535) return PAAC_ERR_ARG;
  if (((uintptr_t)state_in | (uintptr_t)state_out) & 15u) return PAAC_ERR_ARG;
  if ((uintptr_t)newest & 3u) return PAAC_ERR_ARG;
  const cudaError_t launched = launch_overlapped_on((cudaStream_t)stream, stack_push_kernel, dim3(2, n), dim3(SP_THREADS), 0, state_in, newest, restart, state_out);
  return launch_status(launched);
}

extern "C" int paac_preprocess(const uint8_t* raw_prev, const uint8_t* raw_last, const uint8_t* state_in,
                               uint8_t* state_out, int n, void* stream) {
  using namespace paac;
  if (!raw_prev || !raw_last || !state_out || n < 1 || n > 65535) return PAAC_ERR_ARG;
  if (((uintptr_t)raw_prev | (uintptr_t)raw_last) & 15u) return PAAC_ERR_ARG;
  if (((uintptr_t)state_out | (uintptr_t)state_in) & 3u) return PAAC_ERR_ARG;
  // a function's attributes belong to the current device, and this entry point works on any
  static PerDevice<bool> ready;
  int device = -1;
  const bool ok = cudaGetDevice(&device) == cudaSuccess && ready.get(device, [](bool&) {
    return cudaFuncSetAttribute(preprocess_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PpShared)) == cudaSuccess;
  }) != nullptr;
  if (!ok) { cudaGetLastError(); return PAAC_ERR_CUDA; }
  const int tasks = PP_BANDS * n, blocks = tasks < 2 * 148 ? tasks : 2 * 148;      // two blocks per SM are resident
  const cudaError_t launched = launch_overlapped_on((cudaStream_t)stream, preprocess_kernel, dim3(blocks), dim3(PP_THREADS), sizeof(PpShared), raw_prev, raw_last,
                                                    state_in, state_out, tasks);
  return launch_status(launched);
}
