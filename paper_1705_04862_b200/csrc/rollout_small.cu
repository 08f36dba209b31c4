// The forward passes of a whole rollout of the smaller network in one launch, for batches of a few environments.
//
// With 1 to 64 states a step of the layer-by-layer path is four launches of 5 us whose work is a fraction of that.  Here one
// block per SM stays for the rollout and walks its steps.  Environment e belongs to a group of C blocks (C = 16, 8, 4 or
// 2, as many as fit): each computes its share of the first layer's positions, and from the rows that it needs of everybody's its share of
// the second layer's.  The fully connected layer is where the states meet: 21 runs of 128 inputs x 4 tiles of 64 units are
// dealt to 84 blocks, whose weight tile stays in shared memory for the whole rollout, so that each step reads only
// activations.  Every block of a group then finishes its
// environment's state by itself (sum over the runs, heads, draw, transition: the same numbers in each), and writes its
// share of the next frame, of which it keeps the rows its next share of the first layer reads.
//
// Arithmetic is that of the layer-by-layer path to the bit: one chain of fused multiply-adds per output in ascending k,
// 128-long runs of the fully connected layer added in double.
//
// The blocks hand each other both maps and the runs' sums as words that carry their step (step_words.cuh).  A word of a map is overwritten
// for the next step only after all that read it have: a block starts a step with the sums of all runs of the one before, which
// were made from all positions of the second map and they from all rows of the first.  A run's sums, however, need a few positions
// only, whose blocks may be a step ahead of others of their group, so there are two sets of sums, used in turn: those of a step
// are overwritten two steps later, when every block of the group has finished it.
//
// What bounds a step: latency; three hand-overs of about a microsecond and passes that are chains.  With 32 states a step takes 18 us
// (12 with 4): first layer 4.8, second 4.0 (its weights, read from shared memory by every warp), waiting for the second map 1.2 and
// the fully connected runs 3, waiting for their sums 1.0, heads, draw and transition 0.85.  With two barriers over the
// device (1.3 us each, and a second round trip through L2 to read what they guard) instead of words, a rollout of five steps and the
// bootstrap took 84 us with 4 states, 122 with 32 and 205 with 74, with them 78, 119 and 202 (and 7 to 8 less since the set-up loads all at once).
//
// With environments outside, a step is one such launch too: each block fetches the part of the state that it needs (or of the newest
// plane) over the host link and writes its share out; actions and values go straight into pinned memory.
//
// Every wait is bounded: a block that gives up raises the error word and goes on without waiting.
#include <type_traits>

#include "env_device.cuh"
#include "kernels.h"
#include "step_words.cuh"

namespace paac {

constexpr int RS_THREADS = 256, RS_F = 256, RS_IN = 2592, RS_RUN = 128, RS_RUNS = (RS_IN + RS_RUN - 1) / RS_RUN, RS_COLS = 64;
constexpr int RS_TILES = RS_RUNS * (RS_F / RS_COLS), RS_FC_LD = RS_RUN + 4, RS_ROWS = 32;
typedef NipsConv1 RC1;
typedef NipsConv2 RC2;
constexpr int RS_POS1 = RC1::OH * RC1::OW, RS_POS2 = RC2::OH * RC2::OW;        // 400 and 81

struct RsArgs {
  int n, C, A, steps, blocks;             // forward passes: slots t0 .. t0 + steps - 1
  uint32_t t0;
  const uint8_t* frames; size_t frame_step;       // states of slot t0, and from one slot to the next
  uint8_t* next_frames;                           // states of the slot after the last one that steps (rollout)
  int sample_steps;                               // of the passes, so many sample an action (and, with `env`, step it)
  bool env;
  uint4* map1;                                    // words: [n][400][8], two channels each
  uint4* map2;                                    // [n][81][16]
  uint2* sums;                                    // [2][RS_RUNS][n][RS_F], by the step's lowest bit
  uint32_t* sync;
  const float *b1, *b2, *bfc, *bpi, *bv;
  float *logits, *values, *uniforms;
  int32_t *actions, *sampled, *counters;
  const int32_t* forced;
  int8_t* rewards; uint8_t* terminals;
  uint64_t seed; uint64_t* step_base; uint32_t advance;
  uint32_t term_denom; int pattern_actions;
  HeadMode mode;
  HostStep host;
  uint32_t* error_word; uint32_t polls;
};

__device__ __forceinline__ void rs_fma4(float (&acc)[4], float a, const float4 w) {
  acc[0] = fmaf(a, w.x, acc[0]); acc[1] = fmaf(a, w.y, acc[1]); acc[2] = fmaf(a, w.z, acc[2]); acc[3] = fmaf(a, w.w, acc[3]);
}
__device__ __forceinline__ float4 rs_relu(const float (&acc)[4], float scale, const float* b) {
  return make_float4(fmaxf(fmaf(acc[0], scale, b[0]), 0.f), fmaxf(fmaf(acc[1], scale, b[1]), 0.f), fmaxf(fmaf(acc[2], scale, b[2]), 0.f),
                     fmaxf(fmaf(acc[3], scale, b[3]), 0.f));
}
// four neighbouring outputs: as they are stored, and as words with the value the next layer reads
__device__ __forceinline__ float4 rs_stored(const float4 v, const float*) { return v; }
__device__ __forceinline__ float4 rs_stored(const float4 v, const bf16*) {
  return make_float4(to_f(from_f<bf16>(v.x)), to_f(from_f<bf16>(v.y)), to_f(from_f<bf16>(v.z)), to_f(from_f<bf16>(v.w)));
}
template <class T> __device__ __forceinline__ void rs_hand(T* at, uint4* words, const float4 v, uint32_t step) {
  store4(at, v);
  const float4 w = rs_stored(v, at);
  word_store(words, __float_as_uint(w.x), __float_as_uint(w.y), step);
  word_store(words + 1, __float_as_uint(w.z), __float_as_uint(w.w), step);
}

// shared memory, in floats
constexpr int RS_W1 = 0, RS_W2 = RS_W1 + RC1::KK * RC1::CO, RS_FCW = RS_W2 + RC2::KK * RC2::CO, RS_FCA = RS_FCW + RS_COLS * RS_FC_LD,
              RS_ACT1 = RS_FCA + RS_ROWS * RS_FC_LD, RS_FRAME = RS_ACT1 + RS_POS1 * RC1::CO, RS_HEADW = RS_FRAME + FRAME_BYTES / 4;

// First layer: `share` positions from pos0, 4 channels and PP positions (`apart` apart) per thread.  The passes of both
// convolutions are bound by weights going from shared memory to registers (16 floats a thread for four k, whatever PP is),
// so PP is as large as leaves every scheduler one warp.
template <class T, int PP>
__device__ __forceinline__ void rs_conv1(const float* sm, const float* b1, T* act, uint4* words, uint32_t step, int pos0, int share) {
  const int q = threadIdx.x & 3, p = threadIdx.x >> 2, apart = (share + PP - 1) / PP;
  const uint32_t* frame = reinterpret_cast<const uint32_t*>(sm + RS_FRAME);
  const float4* w = reinterpret_cast<const float4*>(sm + RS_W1) + q;                   // [k][16]
  float acc[PP][4];
  int base[PP];
#pragma unroll
  for (int i = 0; i < PP; ++i) {
    const int pos = pos0 + min(p + apart * i, share - 1);
    base[i] = (pos / RC1::OW * RC1::S) * RC1::W + pos % RC1::OW * RC1::S;
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[i][c] = 0.f;
  }
  if (p < apart)
    for (int r = 0; r < RC1::K; ++r) {
#pragma unroll
      for (int s = 0; s < RC1::K; ++s) {
        float4 a[PP];
#pragma unroll
        for (int i = 0; i < PP; ++i) a[i] = widen4(frame[base[i] + r * RC1::W + s]);
        const int k = (r * RC1::K + s) * 4;
        const float4 w0 = w[k * 4], w1 = w[(k + 1) * 4], w2 = w[(k + 2) * 4], w3 = w[(k + 3) * 4];
#pragma unroll
        for (int i = 0; i < PP; ++i) { rs_fma4(acc[i], a[i].x, w0); rs_fma4(acc[i], a[i].y, w1); rs_fma4(acc[i], a[i].z, w2); rs_fma4(acc[i], a[i].w, w3); }
      }
    }
#pragma unroll
  for (int i = 0; i < PP; ++i)
    if (p < apart && p + apart * i < share) {
      const int pos = pos0 + p + apart * i;
      rs_hand(act + (size_t)pos * RC1::CO + 4 * q, words + pos * (RC1::CO / 2) + 2 * q, rs_relu(acc[i], 1.0f / 255.0f, b1 + 4 * q), step);
    }
}
// Second layer: the same with 8 groups of 4 channels, the input rows in shared memory.
template <class T, int PP>
__device__ __forceinline__ void rs_conv2(const float* sm, const float* b2, T* act, uint4* words, uint32_t step, int pos0, int share) {
  const int q = threadIdx.x & 7, p = threadIdx.x >> 3, apart = (share + PP - 1) / PP;
  const float4* in = reinterpret_cast<const float4*>(sm + RS_ACT1);                    // [20][20][16]
  const float4* w = reinterpret_cast<const float4*>(sm + RS_W2) + q;                   // [k][32]
  float acc[PP][4];
  int base[PP];
#pragma unroll
  for (int i = 0; i < PP; ++i) {
    const int pos = pos0 + min(p + apart * i, share - 1);
    base[i] = ((pos / RC2::OW * RC2::S) * RC2::W + pos % RC2::OW * RC2::S) * (RC2::C / 4);
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[i][c] = 0.f;
  }
  if (p < apart)
    for (int r = 0; r < RC2::K; ++r) {
#pragma unroll 4
      for (int sc = 0; sc < RC2::K * RC2::C / 4; ++sc) {                               // (s, four input channels)
        float4 a[PP];
#pragma unroll
        for (int i = 0; i < PP; ++i) a[i] = in[base[i] + r * (RC2::W * RC2::C / 4) + sc];
        const int k = r * RC2::K * RC2::C + sc * 4;
        const float4 w0 = w[k * 8], w1 = w[(k + 1) * 8], w2 = w[(k + 2) * 8], w3 = w[(k + 3) * 8];
#pragma unroll
        for (int i = 0; i < PP; ++i) { rs_fma4(acc[i], a[i].x, w0); rs_fma4(acc[i], a[i].y, w1); rs_fma4(acc[i], a[i].z, w2); rs_fma4(acc[i], a[i].w, w3); }
      }
    }
#pragma unroll
  for (int i = 0; i < PP; ++i)
    if (p < apart && p + apart * i < share) {
      const int pos = pos0 + p + apart * i;
      rs_hand(act + (size_t)pos * RC2::CO + 4 * q, words + pos * (RC2::CO / 2) + 2 * q, rs_relu(acc[i], 1.f, b2 + 4 * q), step);
    }
}

template <class T, class TW, int C>
__global__ void __launch_bounds__(RS_THREADS, 1)
rollout_small_kernel(RsArgs q, const TW* w1, const TW* w2, const TW* wfc, const TW* wpi, const TW* wv, T* act1, T* act2, T* h) {
  extern __shared__ __align__(16) float sm[];
  __shared__ float xs[RS_F], zs[33];
  __shared__ EnvFrame s_frame;
  __shared__ int32_t s_action;
  __shared__ volatile uint32_t s_dead;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n = q.n, A = q.A;
  const bool conv = (int)blockIdx.x < n * C;
  const int e = blockIdx.x / C, rank = blockIdx.x % C;
  const int tile = q.blocks - 1 - (int)blockIdx.x;                 // of the fully connected layer; the last blocks have one each
  const bool fc = tile < RS_TILES;
  const int run = tile / (RS_F / RS_COLS), col0 = tile % (RS_F / RS_COLS) * RS_COLS, k0 = run * RS_RUN;
  const int len = min(RS_RUN, RS_IN - k0);
  constexpr int SHARE1 = RS_POS1 / C, PP1 = C == 16 ? 1 : (C == 8 ? 2 : (C == 4 ? 2 : 7)), PP2 = C == 16 ? 1 : (C == 8 ? 2 : (C == 4 ? 3 : 6));
  static_assert(RS_POS1 % C == 0, "equal shares of the first layer");
  const int pos1 = rank * SHARE1, pos2 = RS_POS2 * rank / C, share2 = RS_POS2 * (rank + 1) / C - pos2;
  const int row_lo = pos1 / RC1::OW * RC1::S, row_hi = (pos1 + SHARE1 - 1) / RC1::OW * RC1::S + RC1::K;      // frame rows read
  constexpr int IN_ROW = RC1::OW * RC1::CO / 4;                    // 16-byte words of a row of the first layer's map
  const int in_lo = pos2 / RC2::OW * RC2::S * IN_ROW, in_hi = ((pos2 + share2 - 1) / RC2::OW * RC2::S + RC2::K) * IN_ROW;
  uint4* frame = reinterpret_cast<uint4*>(sm + RS_FRAME);
  constexpr int QUADS = FRAME_W / 4;                               // 16-byte words of a frame row

  // this block's share of a frame, and the rows of it that its share of the first layer reads
  const int own_lo = FRAME_WORDS / 4 * rank / C, own_hi = FRAME_WORDS / 4 * (rank + 1) / C;
  const int part_lo = min(own_lo, row_lo * QUADS), part_hi = max(own_hi, row_hi * QUADS);
  auto place = [&](uint4* state, int i, const uint4 v) {
    if (i >= own_lo && i < own_hi) state[i] = v;
    if (i >= row_lo * QUADS && i < row_hi * QUADS) frame[i] = v;
  };
  // What stays for the rollout: both convolutions' weights as [k][channel], the weight tile, the head weights.  All are asked for before any is
  // used, and what comes over the host link after them, so that one latency covers them all.  (A warp's lanes take a channel each, so
  // that their values go to different banks; value by value in the order of the arrays, the stores of the second layer's weights alone met 32
  // conflicts each: a launch took 8 us more; an iteration at 4 environments 121.7 -> 114.7 us, with whole states of 32 from outside 490 -> 439.)
  constexpr int W1_PER = RC1::KK * RC1::CO / 4 / RS_THREADS, W2_PER = RC2::KK * RC2::CO / 4 / RS_THREADS, FC_PER = RS_COLS * RS_RUN / 4 / RS_THREADS, HEAD_PER = 32 * RS_F / 4 / RS_THREADS;
  const uint32_t epoch = q.sync[0];
  const uint64_t step0 = *q.step_base + q.t0;
  float4 v1[W1_PER], v2[W2_PER], vf[FC_PER], vh[HEAD_PER];
  float value_head = 0.f;
  if (conv) {
#pragma unroll
    for (int u = 0; u < W1_PER; ++u) { const int i = tid + u * RS_THREADS; v1[u] = load4(w1 + i % RC1::CO * RC1::KK + i / RC1::CO * 4); }
#pragma unroll
    for (int u = 0; u < W2_PER; ++u) { const int i = tid + u * RS_THREADS; v2[u] = load4(w2 + i % RC2::CO * RC2::KK + i / RC2::CO * 4); }
#pragma unroll
    for (int u = 0; u < HEAD_PER; ++u) { const int i = tid + u * RS_THREADS; if (i < A * RS_F / 4) vh[u] = load4(wpi + 4 * i); }
    if (tid < RS_F) value_head = to_f(wv[tid]);
  }
  if (fc) {
#pragma unroll
    for (int u = 0; u < FC_PER; ++u) {
      const int i = tid + u * RS_THREADS, c = i / (RS_RUN / 4), k = i % (RS_RUN / 4) * 4;
      vf[u] = k < len ? load4(wfc + (size_t)(col0 + c) * RS_IN + k0 + k) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  uint4* const state = reinterpret_cast<uint4*>(const_cast<uint8_t*>(q.frames) + (size_t)e * FRAME_BYTES);
  // the whole state over the host link, or the newest plane, sixteen pixels to a word
  constexpr int MOST = (FRAME_WORDS / 4 + RS_THREADS - 1) / RS_THREADS, MOST_PLANE = (STACK_ITEMS + RS_THREADS - 1) / RS_THREADS;
  static_assert(MOST_PLANE <= MOST, "the same registers");
  uint4 in[MOST];
  if (conv && q.host.states != nullptr) {
    const uint4* src = reinterpret_cast<const uint4*>(q.host.states) + (size_t)e * (FRAME_WORDS / 4);
#pragma unroll
    for (int u = 0; u < MOST; ++u)
      if (part_lo + tid + u * RS_THREADS < part_hi) in[u] = src[part_lo + tid + u * RS_THREADS];
  } else if (conv && q.host.newest != nullptr) {
    const uint4* src = reinterpret_cast<const uint4*>(q.host.newest) + (size_t)e * STACK_ITEMS;
#pragma unroll
    for (int u = 0; u < MOST_PLANE; ++u)
      if (part_lo / 4 + tid + u * RS_THREADS < (part_hi + 3) / 4) in[u] = src[part_lo / 4 + tid + u * RS_THREADS];
  } else if (conv) {
#pragma unroll
    for (int u = 0; u < MOST; ++u)
      if (row_lo * QUADS + tid + u * RS_THREADS < row_hi * QUADS) in[u] = __ldcg(state + row_lo * QUADS + tid + u * RS_THREADS);
  }
  if (conv) {
#pragma unroll
    for (int u = 0; u < W1_PER; ++u) {
      float* to = sm + RS_W1 + (tid + u * RS_THREADS) / RC1::CO * 4 * RC1::CO + (tid + u * RS_THREADS) % RC1::CO;
      to[0] = v1[u].x; to[RC1::CO] = v1[u].y; to[2 * RC1::CO] = v1[u].z; to[3 * RC1::CO] = v1[u].w;
    }
#pragma unroll
    for (int u = 0; u < W2_PER; ++u) {
      float* to = sm + RS_W2 + (tid + u * RS_THREADS) / RC2::CO * 4 * RC2::CO + (tid + u * RS_THREADS) % RC2::CO;
      to[0] = v2[u].x; to[RC2::CO] = v2[u].y; to[2 * RC2::CO] = v2[u].z; to[3 * RC2::CO] = v2[u].w;
    }
#pragma unroll
    for (int u = 0; u < HEAD_PER; ++u)
      if (tid + u * RS_THREADS < A * RS_F / 4) *reinterpret_cast<float4*>(sm + RS_HEADW + 4 * (tid + u * RS_THREADS)) = vh[u];
    if (tid < RS_F) sm[RS_HEADW + A * RS_F + tid] = value_head;
  }
  if (fc) {
#pragma unroll
    for (int u = 0; u < FC_PER; ++u) {
      const int i = tid + u * RS_THREADS;
      *reinterpret_cast<float4*>(sm + RS_FCW + i / (RS_RUN / 4) * RS_FC_LD + i % (RS_RUN / 4) * 4) = vf[u];
    }
  }
  if (conv && q.host.states != nullptr) {
#pragma unroll
    for (int u = 0; u < MOST; ++u)
      if (part_lo + tid + u * RS_THREADS < part_hi) place(state, part_lo + tid + u * RS_THREADS, in[u]);
  } else if (conv && q.host.newest != nullptr) {
    // onto the stack of the state before
    const uint4* prev = reinterpret_cast<const uint4*>(q.host.prev) + (size_t)e * (FRAME_WORDS / 4);
    const bool fresh = (q.host.fresh[e >> 5] >> (e & 31)) & 1u;
#pragma unroll
    for (int u = 0; u < MOST_PLANE; ++u) {
      const int i = part_lo / 4 + tid + u * RS_THREADS;
      if (i < (part_hi + 3) / 4) {
        uint4 o[4];
        stack_sixteen(in[u], fresh, prev + 4 * i, o);
#pragma unroll
        for (int k = 0; k < 4; ++k) place(state, 4 * i + k, o[k]);
      }
    }
  } else if (conv) {
#pragma unroll
    for (int u = 0; u < MOST; ++u)
      if (row_lo * QUADS + tid + u * RS_THREADS < row_hi * QUADS) frame[row_lo * QUADS + tid + u * RS_THREADS] = in[u];
  }
  if (tid == 0) s_dead = 0u;
  __syncthreads();

  for (int t = 0; t < q.steps; ++t) {
    const size_t slot = (size_t)t * n;
    const uint32_t tag = epoch + 1u + (uint32_t)t;
    uint2* sums = q.sums + (size_t)(tag & 1u) * RS_RUNS * n * RS_F;
    if (conv) {
      T* a1 = act1 + (slot + e) * RC1::OUT_SIZE;
      T* a2 = act2 + (slot + e) * RC2::OUT_SIZE;
      rs_conv1<T, PP1>(sm, q.b1, a1, q.map1 + (size_t)e * (RS_POS1 * RC1::CO / 2), tag, pos1, SHARE1);
      {
        constexpr int MOST = 8;                    // 16-byte words, two values each: at most twelve rows (C = 2)
        const uint4* src = q.map1 + (size_t)e * (RS_POS1 * RC1::CO / 2) + 2 * in_lo + tid;
        const int count = (2 * (in_hi - in_lo) - tid + RS_THREADS - 1) / RS_THREADS;
        uint4 v[MOST];
        word_await(v, src, RS_THREADS, count, tag, &s_dead, q.error_word, q.polls);
#pragma unroll
        for (int u = 0; u < MOST; ++u)
          if (u < count) reinterpret_cast<float2*>(sm + RS_ACT1)[2 * in_lo + tid + u * RS_THREADS] = make_float2(__uint_as_float(v[u].x), __uint_as_float(v[u].z));
      }
      __syncthreads();
      rs_conv2<T, PP2>(sm, q.b2, a2, q.map2 + (size_t)e * (RS_IN / 2), tag, pos2, share2);
    }
    if (fc) {
      for (int r0 = 0; r0 < n; r0 += RS_ROWS) {
        const int rows = min(RS_ROWS, n - r0);
        if (r0 > 0) __syncthreads();
        {
          // 64 words (two inputs each) to a row of a whole run, 16 to one of the last
          const int per = len / 2, r = tid / per, u = tid % per, apart = RS_THREADS / per, count = (rows - r + apart - 1) / apart;
          const uint4* src = q.map2 + (size_t)(r0 + r) * (RS_IN / 2) + k0 / 2 + u;
          uint4 v[RS_ROWS / 4];
          word_await(v, src, (size_t)apart * (RS_IN / 2), count, tag, &s_dead, q.error_word, q.polls);
#pragma unroll
          for (int i = 0; i < RS_ROWS / 4; ++i)
            if (i < count) *reinterpret_cast<float2*>(sm + RS_FCA + (r + apart * i) * RS_FC_LD + 2 * u) = make_float2(__uint_as_float(v[i].x), __uint_as_float(v[i].z));
        }
        __syncthreads();
        const int cx = tid & 15, ry = tid >> 4;
        const float* pa = sm + RS_FCA + ry * RS_FC_LD;
        const float* pb = sm + RS_FCW + cx * RS_FC_LD;
        float acc[2][4] = {};
        auto columns = [&](auto two_rows) {
          constexpr int R = decltype(two_rows)::value;
#pragma unroll 4
          for (int k = 0; k < len; k += 4) {
            float4 a[R], b[4];
#pragma unroll
            for (int i = 0; i < R; ++i) a[i] = *reinterpret_cast<const float4*>(pa + i * 16 * RS_FC_LD + k);
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = *reinterpret_cast<const float4*>(pb + j * 16 * RS_FC_LD + k);
#pragma unroll
            for (int i = 0; i < R; ++i)
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                acc[i][j] = fmaf(a[i].x, b[j].x, acc[i][j]); acc[i][j] = fmaf(a[i].y, b[j].y, acc[i][j]);
                acc[i][j] = fmaf(a[i].z, b[j].z, acc[i][j]); acc[i][j] = fmaf(a[i].w, b[j].w, acc[i][j]);
              }
          }
        };
        if (ry < rows) { if (rows > 16) columns(std::integral_constant<int, 2>{}); else columns(std::integral_constant<int, 1>{}); }
#pragma unroll
        for (int i = 0; i < 2; ++i)
          if (ry + 16 * i < rows)
#pragma unroll
            for (int j = 0; j < 4; ++j) word_store(sums + ((size_t)run * n + r0 + ry + 16 * i) * RS_F + col0 + cx + 16 * j, __float_as_uint(acc[i][j]), tag);
      }
    }
    if (!conv) continue;
    // ---- the end of the state's pass, in every block of the group ----
    const bool sample = t < q.sample_steps, stepping = sample && q.env;
    EnvPrep prep{};
    if (stepping && tid == 32) prep = env_prepare(q.seed, (uint32_t)e, n, (uint32_t)step0 + t, rank == 0 ? q.counters : nullptr);
    {
      uint2 v[RS_RUNS];
      word_await(v, sums + (size_t)e * RS_F + tid, (size_t)n * RS_F, RS_RUNS, tag, &s_dead, q.error_word, q.polls);
      double s = 0.0;
#pragma unroll
      for (int p = 0; p < RS_RUNS; ++p) s += (double)__uint_as_float(v[p].x);
      const T x = from_f<T>(fmaxf((float)(s + (double)q.bfc[tid]), 0.f));
      if (rank == 0) h[(slot + e) * RS_F + tid] = x;
      xs[tid] = to_f(x);
    }
    __syncthreads();
    for (int k = warp; k <= A; k += RS_THREADS / 32) {
      float acc = 0.f;
#pragma unroll
      for (int i = 0; i < RS_F / 32; ++i) {
        const int at = sizeof(T) == 2 ? lane * (RS_F / 32) + i : lane + 32 * i;
        acc = fmaf(sm[RS_HEADW + k * RS_F + at], xs[at], acc);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane == 0) zs[k] = acc + (k < A ? q.bpi[k] : q.bv[0]);
    }
    __syncthreads();
    if (warp == 0) {
      const int32_t a = warp_finish_heads(q.mode, lane < A ? zs[lane] : -INFINITY, zs[A], lane, A, (size_t)e, q.logits + slot * A, q.values + slot,
                                          sample, q.seed, step0 + t, q.forced ? q.forced + slot : nullptr, q.actions + slot, q.sampled + slot,
                                          q.uniforms + slot);
      if (lane == 0) s_action = a;
      if (q.host.done != nullptr && rank == 0 && lane == 0) {
        if (sample) q.host.actions[e] = a;
        q.host.values[e] = q.values[slot + e];
        __threadfence_system();
      }
    }
    if (!stepping) { __syncthreads(); continue; }
    __syncthreads();
    EnvOutcome o{0, false, 0u};
    if (tid == 32) {
      o = env_outcome(prep, s_action, q.term_denom, q.pattern_actions);
      s_frame = env_frame_of(prep.pre_next, o.tag, q.pattern_actions);
    }
    __syncthreads();
    if (tid == 32 && rank == 0) env_record(prep, o, (uint32_t)e, n, q.rewards + slot, q.terminals + slot, q.counters);
    const EnvFrame f = s_frame;
    // this block's share of the frame for everyone, and the rows it will read itself
    uint8_t* states = t + 1 < q.sample_steps ? const_cast<uint8_t*>(q.frames) + (size_t)(t + 1) * q.frame_step : q.next_frames;
    uint4* out = reinterpret_cast<uint4*>(states + (size_t)e * FRAME_BYTES);
    for (int i = part_lo + tid; i < part_hi; i += RS_THREADS) place(out, i, env_frame_quad(f, (uint32_t)i, q.pattern_actions));
    __syncthreads();
  }
  // Every block has read the counts when the last one ends.
  if (tid == 0) {
    __threadfence();
    if (atomicAdd(q.sync + 1, 1u) == gridDim.x - 1) {
      q.sync[0] = epoch + (uint32_t)q.steps;
      q.sync[1] = 0u;
      if (q.advance) *q.step_base += q.advance;
      if (q.host.done != nullptr) { __threadfence_system(); *q.host.done = 1u; }
    }
  }
}

// Blocks per environment: as many of 16, 8, 4, 2 as leave each a multiprocessor of its own; 0: use the layer-by-layer path.
static int rs_blocks_per_env(int n) { return n <= 9 ? 16 : (n <= 18 ? 8 : (n <= 37 ? 4 : (n <= 74 ? 2 : 0))); }
// One block per SM of a whole device; shared memory up to the largest head.
constexpr int RS_BLOCKS = 148;
static size_t rs_smem(int A) { return (size_t)(RS_HEADW + (A + 1) * RS_F) * sizeof(float); }

template <class T_, int C> struct RsKernel {
  typedef T_ T;                                        // storage of weights and activations
  static auto kernel() { return rollout_small_kernel<T, T, C>; }
  // Blocks that wait for one another all have to be resident: what a cooperative launch checks, asked for beforehand so that
  // a device with fewer multiprocessors, or a build that takes more registers, goes layer by layer instead of failing.
  static bool fits() {
    static const bool resident = [] {
      int dev = 0, sms = 0, coop = 0, per_sm = 0;
      const int smem = (int)rs_smem(32);
      const bool known = cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
                         cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess &&
                         cudaFuncSetAttribute(kernel(), cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess &&
                         cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel(), RS_THREADS, smem) == cudaSuccess;
      if (!known) cudaGetLastError();
      return known && coop != 0 && per_sm * sms >= RS_BLOCKS;
    }();
    return resident;
  }
};
template <class F> static auto rs_pick(int prec, int C, F f) {
  auto of = [&](auto t) {
    typedef decltype(t) T;
    if (C == 16) return f(RsKernel<T, 16>{});
    if (C == 8) return f(RsKernel<T, 8>{});
    if (C == 4) return f(RsKernel<T, 4>{});
    return f(RsKernel<T, 2>{});
  };
  return prec == PAAC_BF16 ? of(bf16{}) : of(float{});
}

bool rollout_small_supported(const LaunchCtx& lc, int arch, int prec, int n) {
  const int C = rs_blocks_per_env(n);
  return arch == PAAC_ARCH_NIPS && !lc.fp32_tensor_cores && C != 0 && rs_pick(prec, C, [](auto k) { return k.fits(); });
}
// of 16 bytes: both maps, and two sets of the runs' sums at two to a word
static size_t rs_map1_words(int n) { return (size_t)n * RS_POS1 * RC1::CO / 2; }
static size_t rs_map2_words(int n) { return (size_t)n * RS_IN / 2; }
size_t rollout_small_words(int n) { return rs_blocks_per_env(n) == 0 ? 0 : rs_map1_words(n) + rs_map2_words(n) + (size_t)n * RS_RUNS * RS_F; }

void launch_rollout_small(LaunchCtx& lc, int prec, const NetDims& nd, const float* theta, const bf16* theta16, const SmallRollout& r) {
  const LayerDims* d = nd.layer;
  RsArgs q{};
  q.n = r.n; q.C = rs_blocks_per_env(r.n); q.A = nd.A; q.steps = r.steps; q.blocks = RS_BLOCKS; q.t0 = r.t0;
  q.frames = r.frames; q.frame_step = r.frame_step; q.next_frames = r.env.next_frames; q.sample_steps = r.sample_steps; q.env = r.step_env;
  q.map1 = (uint4*)r.words; q.map2 = q.map1 + rs_map1_words(r.n); q.sums = (uint2*)(q.map2 + rs_map2_words(r.n)); q.sync = r.sync; q.host = r.host;
  q.b1 = theta + d[0].b_off; q.b2 = theta + d[1].b_off; q.bfc = theta + d[2].b_off; q.bpi = theta + nd.pi_b; q.bv = theta + nd.v_b;
  q.logits = r.logits; q.values = r.values; q.uniforms = r.uniforms; q.actions = r.actions; q.sampled = r.sampled; q.counters = r.env.counters;
  q.forced = r.forced; q.rewards = r.env.rewards; q.terminals = r.env.terminals; q.seed = r.seed; q.step_base = r.step_base; q.advance = r.advance;
  q.term_denom = r.env.term_denom; q.pattern_actions = r.env.pattern_actions; q.mode = r.mode;
  q.error_word = r.error_word; q.polls = r.polls;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(q.blocks); cfg.blockDim = dim3(RS_THREADS); cfg.dynamicSmemBytes = rs_smem(q.A); cfg.stream = lc.st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative; attr[0].val.cooperative = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  lc.serialize_next = false;
  KernelScope scope(lc, KID_SMALL_ROLLOUT);
  const bool launched = rs_pick(prec, q.C, [&](auto k) {
    typedef typename decltype(k)::T T;
    const T* w;
    if constexpr (sizeof(T) == 2) w = theta16; else w = theta;
    return k.fits() && cudaLaunchKernelEx(&cfg, k.kernel(), q, w + d[0].w_off, w + d[1].w_off, w + d[2].w_off, w + nd.pi_w, w + nd.v_w,
                                          (T*)r.act[0], (T*)r.act[1], (T*)r.act[2]) == cudaSuccess;
  });
  if (!launched) lc.host_failure = true;
}

}  // namespace paac
