// The forward passes of a whole rollout of the larger network (bf16) in one launch, for batches that leave the device idle.
//
// Layer by layer, a step of 32 states is five launches of about 4 us (set-up, first operands, last tile) for two
// microseconds of work.  Here one block per SM stays for the rollout.  An environment belongs to a cluster of C blocks: each
// holds the whole frame and its share of the channels of every convolution's weights, and hands its channels of the first two
// layers' maps to the others as one bulk copy each through distributed shared memory (stores to another block's shared
// memory, a few bytes each, took over a microsecond a layer).  The fully connected layer is where the states meet: its
// 8 slices of K x 16 tiles of 32 units are dealt to 128 blocks, whose weights stay in shared memory for the rollout.  States
// reach them, and their sums reach the environments' blocks, as words that carry the number of the step beside the
// value: a reader polls the word itself, so no barrier over the device and no second round trip through L2 is needed.  Each
// block of a cluster then finishes its share of the hidden units and heads, all take the action, and each makes the
// next frame for itself and writes its share of it out.
//
// Why mma.sync here and not tcgen05: a block's share of a layer is 49 to 400 rows by 8 to 32 channels, a few hundred
// m16n8k16 instructions.  They take their operands from shared memory as they lie (the first layer's straight from the
// frame's bytes) and leave their results in registers, where a tensor-memory accumulator costs a commit, a wait and a
// read-back of about a microsecond per layer, as much as the multiplying.  Both instructions add sixteen products and the
// accumulator in the same way, so the numbers are those of the layer-by-layer path to the bit: the same groups of
// sixteen k in the same order (the first layer's depend on the parity of the position, the second and third keep the two sums of
// tc_shift_t_kernel, the fully connected layer its eight slices, the heads their tree).
//
// A word (step_words.cuh) of a step is overwritten by the next step only after everything that reads it has: an environment's
// blocks start a step with the sums of the one before, which the fully connected blocks made from those words.
//
// With environments outside, a step is one such launch too: while the weights come in, each block of a cluster fetches its share of the
// environment's newest plane over the host link and writes its share of the state, and the environment's action and value go straight
// into pinned memory, the flag behind them set by the block that ends last.  Where the planes lie and which stacks start afresh are
// launch arguments: read from pinned memory by every block, they took 16 us each (reads of one address are served one after
// the other).
//
// Every wait is bounded.  A block that gave up finishes its step without waiting (it arrives at each of its barriers once a step, so
// none is told of more bytes than it can count) and leaves the loop.  The blocks of its cluster then linger together: nobody leaves
// before what was sent to or from it can have arrived.
#include <cuda_fp16.h>

#include "env_device.cuh"
#include "kernels.h"
#include "step_words.cuh"

namespace paac {

typedef NatConv1 TC1; typedef NatConv2 TC2; typedef NatConv3 TC3;
constexpr int RT_THREADS = 512, RT_WARPS = RT_THREADS / 32;
constexpr int RT_F = 512, RT_SLICES = 8, RT_TILE = 32, RT_FC_BLOCKS = RT_SLICES * (RT_F / RT_TILE), RT_ROWS = 64;
constexpr int RT_POS3 = TC3::OH * TC3::OW, RT_FC_LD = 7 * 128;                      // 49 blocks of 64 k, six or seven to a slice

struct RtArgs {
  int n, A, steps;                                // forward passes: slots t0 .. t0 + steps - 1
  uint32_t t0;
  const uint8_t* frames; size_t frame_step;       // states of slot t0, and from one slot to the next
  uint8_t* next_frames;                           // states of the slot after the last one that steps (rollout)
  int sample_steps;                               // of the passes, so many sample an action (and, with `env`, step it)
  bool env;
  const __half* w1;                               // [co][tap][py][16], times 2^8
  const bf16 *w2, *w3, *wfc, *wpi, *wv;
  const float *b1, *b2, *b3, *bfc, *bpi, *bv;
  float scale1;                                   // of the first layer's sums
  bf16 *act1, *act2, *act3, *h;
  uint4* maps;                                    // [n][49][16]: third layer's outputs, four channels to a word pair
  uint4* sums;                                    // [8][n][256]: fully connected sums of a slice, two units to a word pair
  uint32_t* sync;                                 // steps so far, blocks that have ended
  float *logits, *values, *uniforms;
  int32_t *actions, *sampled, *counters;
  const int32_t* forced;
  int8_t* rewards; uint8_t* terminals;
  uint64_t seed; uint64_t* step_base; uint32_t advance;
  uint32_t term_denom; int pattern_actions;
  HeadMode mode;
  HostStep host;                                  // external environments (one pass)
  uint32_t* error_word; uint32_t polls;
};

// ---- instructions ------------------------------------------------------------------------------------------------------
__device__ __forceinline__ void rt_ldsm4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void rt_mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void rt_mma_f16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t rt_relu_pack(float lo, float hi) {          // ReLU and the bf16 rounding
  uint32_t r;
  asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
__device__ __forceinline__ uint32_t rt_rank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ uint32_t rt_map(uint32_t addr, uint32_t rank) {      // the same shared address in block `rank` of the cluster
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
template <int BYTES> __device__ __forceinline__ void rt_copy_async(uint32_t to, const void* from) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(to), "l"(from), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void rt_sts(uint32_t addr, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }
__device__ __forceinline__ void rt_store(uint32_t to, uint32_t v) { asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(to), "r"(v) : "memory"); }
// four bytes, or `bytes` of this block's shared memory, to another block's, counted at its barrier
__device__ __forceinline__ void rt_send(uint32_t to, uint32_t v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.u32 [%0], %1, [%2];" ::"r"(to), "r"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ void rt_send_bulk(uint32_t to, uint32_t from, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(to), "r"(from), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void rt_cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void rt_pair_sync(int id) {                          // two warps
  __syncwarp();
  asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory");
}

// Shared memory, in bytes.  Rows of weights are in groups of 128 bytes whose 16-byte pieces are permuted by the row's low bits, so
// that eight rows of a fragment lie in different banks.  The maps are planes of eight channels, 16 bytes per position, so that a
// block's channels are one piece to send.  A fragment's rows are neighbouring positions of the next layer's map: the first layer's
// positions are ordered (y mod 2, y / 2, x mod 2, x / 2), as the second layer's window moves by two, and rows are 25 and 15
// places apart, so that the step from the end of a row of 9 or 7 to the next is one place more, modulo eight (with rows packed
// 60 % of the fragments met a bank conflict and the second layer took 1.07 instead of 0.85 us).
constexpr int RT_ROW1 = 25, RT_ROW2 = 15, RT_PLANE1 = 20 * RT_ROW1 * 16 + 16, RT_PLANE2 = (9 * RT_ROW2 + 1) * 16;
__device__ __forceinline__ int rt_place1(int y, int x) { return ((y & 1) * 10 + (y >> 1)) * RT_ROW1 + (x & 1) * 10 + (x >> 1); }
template <int C> struct RtMem {
  static constexpr int N1 = 4 / C, N2 = 8 / C, COLS = RT_F / C, RUNS = 32 / C;     // 8-channel tiles of the layers; units and running sums of a block
  static constexpr int W1 = 0, W2 = W1 + N1 * 4096, W3 = W2 + N2 * 8 * 1024, WFC = W3 + N2 * 8 * 1152, HEADW = WFC + RT_TILE * RT_FC_LD,
                       FRAME = HEADW + (33 * COLS * 2 + 127) / 128 * 128, ACT1 = FRAME + (FRAME_BYTES + 127) / 128 * 128, ACT2 = ACT1 + (4 * RT_PLANE1 + 127) / 128 * 128,
                       B1 = ACT2 + (8 * RT_PLANE2 + 127) / 128 * 128, B2 = B1 + N1 * 32, B3 = B2 + N2 * 32, BFC = B3 + N2 * 32, BHEAD = BFC + COLS * 4,
                       XS = (BHEAD + 33 * 4 + 15) / 16 * 16, ZS = XS + COLS * 4, TOTAL = ZS + C * 36 * 4;
  static constexpr int ROWS = FRAME;              // the states' rows for the fully connected layer lie over the frame and the maps
  static_assert(ROWS + RT_ROWS * RT_FC_LD <= B1, "rows of the fully connected layer");
  static_assert(TOTAL <= 227 * 1024, "shared memory");
};

// First layer, this block's channels of all 400 positions.  Positions come in tiles of
// sixteen of one parity (of e + y + x), as the order in which tc_conv1_kernel adds the four block taps depends on it; eight
// neighbouring ones lie in two rows, so that their bytes come from different banks.  A warp takes a tile of either parity.
template <int C>
__device__ __forceinline__ void rt_conv1(const uint8_t* smem, uint32_t sm, const RtArgs& q, int e, int rank, int tile, int lane) {
  typedef RtMem<C> S;
  const int g = lane >> 2, t = lane & 3;
  int y[2], x[2][2];
  const uint8_t* at[2][2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int p = min(tile * 16 + g + 8 * i, 199), pair = p / 20, r = p - 20 * pair;
    y[i] = 2 * pair + (r & 1);
#pragma unroll
    for (int odd = 0; odd < 2; ++odd) {
      x[odd][i] = (r & ~1) + ((odd + e + y[i]) & 1);
      at[odd][i] = smem + S::FRAME + y[i] * 4 * (FRAME_W * 4) + x[odd][i] * 16 + 4 * t;
    }
  }
  float acc[2][S::N1][4];
#pragma unroll
  for (int odd = 0; odd < 2; ++odd)
#pragma unroll
    for (int j = 0; j < S::N1; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[odd][j][i] = 0.f;
  const uint2* w = reinterpret_cast<const uint2*>(smem + S::W1) + lane;
#pragma unroll
  for (int up = 0; up < 2; ++up) {
    uint2 b[2][4][S::N1];                                           // the two taps of a row of blocks
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int py = 0; py < 4; ++py)
#pragma unroll
        for (int j = 0; j < S::N1; ++j) b[r][py][j] = w[(j * 16 + (2 * up + r) * 4 + py) * 32];
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int py = 0; py < 4; ++py)
#pragma unroll
        for (int odd = 0; odd < 2; ++odd) {
          const int r = up == 0 && !odd ? 1 - k : k;                // even positions: the right block of the upper pair first
          const int off = up * (4 * FRAME_W * 4) + r * 16 + py * (FRAME_W * 4);
          const uint32_t v0 = *reinterpret_cast<const uint32_t*>(at[odd][0] + off), v1 = *reinterpret_cast<const uint32_t*>(at[odd][1] + off);
          // a byte in the low half of a 16-bit word is the fp16 value n 2^-24 (see u8x4_to_f16x4)
          const uint32_t a[4] = {__byte_perm(v0, 0u, 0x4140), __byte_perm(v1, 0u, 0x4140), __byte_perm(v0, 0u, 0x4342), __byte_perm(v1, 0u, 0x4342)};
#pragma unroll
          for (int j = 0; j < S::N1; ++j) rt_mma_f16(acc[odd][j], a, b[r][py][j].x, b[r][py][j].y);
        }
  }
#pragma unroll
  for (int j = 0; j < S::N1; ++j) {
    const int nt = rank * S::N1 + j;
    const float2 b = *reinterpret_cast<const float2*>(smem + S::B1 + (j * 8 + 2 * t) * 4);
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (tile * 16 + g + 8 * i < 200)
#pragma unroll
        for (int odd = 0; odd < 2; ++odd) {
          const float* s = acc[odd][j] + 2 * i;
          const __nv_bfloat162 v = __floats2bfloat162_rn(fmaxf(fmaf(s[0], q.scale1, b.x), 0.f), fmaxf(fmaf(s[1], q.scale1, b.y), 0.f));
          rt_sts(sm + S::ACT1 + nt * RT_PLANE1 + rt_place1(y[i], x[odd][i]) * 16 + 4 * t, *reinterpret_cast<const uint32_t*>(&v));
        }
  }
}

// One of the two sums of the second or third layer (see tc_shift_t_kernel): MT tiles of sixteen positions (at(tile, step): where this
// lane's eight channels of its position's input lie), NT tiles of eight channels, taps in the order given.  An instruction's operands come from shared memory
// at 128 bytes a clock, 512 for A and 256 for B: MT x NT tiles to a warp divide that, and fragments are asked for two steps of
// sixteen k ahead.
template <int MT, int NT, int TAPS, class At, class TapOf>
__device__ __forceinline__ void rt_chain(float (&acc)[MT][NT][4], uint32_t w, int w_ld, int lane, At at, TapOf tap_of) {
  static_assert(NT % 2 == 0, "a load brings B for two tiles");
  const uint32_t bhalf = ((uint32_t)lane >> 3) & 1u;
  const uint32_t brow = (uint32_t)((lane & 7) + (lane >> 4) * 8), bsw = brow & 7u, bbase = w + brow * w_ld;
#pragma unroll
  for (int m = 0; m < MT; ++m)
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[m][j][i] = 0.f;
  uint32_t a[3][MT][4], b[3][NT / 2][4];
  auto load = [&](int step, int into) {
    const int i = step >> 2, kk = step & 3;
#pragma unroll
    for (int m = 0; m < MT; ++m) rt_ldsm4(at(m, i, kk), a[into][m]);
#pragma unroll
    for (int j = 0; j < NT / 2; ++j) rt_ldsm4(bbase + j * 16 * w_ld + (((uint32_t)tap_of(i) * 8u + 2u * kk + bhalf) ^ bsw) * 16u, b[into][j]);
  };
  load(0, 0);
  load(1, 1);
#pragma unroll
  for (int step = 0; step < 4 * TAPS; ++step) {
    if (step + 2 < 4 * TAPS) load(step + 2, (step + 2) % 3);
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
      for (int j = 0; j < NT; ++j) rt_mma_bf16(acc[m][j], a[step % 3][m], b[step % 3][j / 2][2 * (j & 1)], b[step % 3][j / 2][2 * (j & 1) + 1]);
  }
}

// (The cluster's size is part of the kernel: launched with a cluster attribute instead it runs as well, but not under a profiler,
// where the launch failed as soon as the blocks sent each other bulk copies.)
template <int C>
__global__ void __cluster_dims__(C, 1, 1) __launch_bounds__(RT_THREADS, 1)
rollout_tc_kernel(const __grid_constant__ RtArgs q) {
  typedef RtMem<C> S;
  extern __shared__ __align__(128) uint8_t rt_smem[];
  __shared__ EnvFrame s_frame;
  __shared__ EnvPrep s_prep;
  __shared__ volatile uint32_t s_dead, s_linger;                  // a wait here, or in a block of the cluster, gave up
  __shared__ __align__(8) uint64_t s_map1, s_map2, s_heads;       // the other blocks' shares have arrived
  const uint32_t sm = tc::smem_u32(rt_smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n = q.n, A = q.A;
  const int g = lane >> 2, t4 = lane & 3;
  const int rank = (int)rt_rank(), e = blockIdx.x / C;             // this cluster's environment
  const bool conv = e < n;
  const bool fc = blockIdx.x < RT_FC_BLOCKS;
  const int slice = blockIdx.x % RT_SLICES, unit0 = blockIdx.x / RT_SLICES * RT_TILE;
  const int kb0 = slice * 6 + (slice > 0 ? 1 : 0), kbs = slice == 0 ? 7 : 6;           // 49 blocks of 64 k: seven, then six each
  // this block's share of the hidden units: column (j, run, i) is unit half 256 + 64 j + 4 (run STEP + low) + i, whole subtrees
  // of the heads' sums (see tc_fc_cluster_kernel)
  constexpr int STEP = C / 2;
  const int half = rank / STEP, low = rank % STEP;
  auto unit_of = [&](int col) { return half * 256 + 64 * (col / (4 * S::RUNS)) + 4 * ((col / 4 % S::RUNS) * STEP + low) + (col & 3); };

  // the newest plane comes over the host link meanwhile: sixteen pixels to a thread
  const int px_lo = STACK_ITEMS * rank / C, px_hi = STACK_ITEMS * (rank + 1) / C;
  static_assert((STACK_ITEMS + C - 1) / C <= RT_THREADS && FRAME_WORDS / 4 / C <= 2 * RT_THREADS, "one piece to a thread");
  uint4 plane{};
  const bool pulls = q.host.newest != nullptr && conv && px_lo + tid < px_hi;
  if (pulls) plane = reinterpret_cast<const uint4*>(q.host.newest)[(size_t)e * STACK_ITEMS + px_lo + tid];
  // or the whole state: four such words
  const int st_lo = FRAME_WORDS / 4 * rank / C, st_hi = FRAME_WORDS / 4 * (rank + 1) / C;
  uint4 whole[2];
  if (q.host.states != nullptr && conv)
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (st_lo + tid + i * RT_THREADS < st_hi) whole[i] = reinterpret_cast<const uint4*>(q.host.states)[(size_t)e * (FRAME_WORDS / 4) + st_lo + tid + i * RT_THREADS];

  // ---- what stays for the rollout ----
  // Everything by asynchronous copies, so that one latency covers all of it: with the small arrays loaded and stored by hand, one after
  // the other, this took 2.7 us (a rollout at 32 environments 74.5 us; an iteration 150.0, now 148.0; with environments outside, six such launches,
  // the iterations of one run differ by more).
  const uint32_t epoch = q.sync[0];
  if (tid == 0) {
    s_dead = 0u; s_linger = 0u;
    tc::mbar_init(&s_map1, 1); tc::mbar_init(&s_map2, 1); tc::mbar_init(&s_heads, 1);
    tc::fence_barrier_init();
  }
  if (conv) {
    for (int i = tid; i < S::N1 * 16 * 32; i += RT_THREADS) {
      const int l = i & 31, step = i >> 5, j = step >> 4, co = (rank * S::N1 + j) * 8 + (l >> 2);
      rt_copy_async<8>(sm + S::W1 + i * 8, q.w1 + ((size_t)co * 16 + (step & 15)) * 16 + 4 * (l & 3));
    }
    for (int i = tid; i < S::N2 * 8 * 64; i += RT_THREADS) {
      const uint32_t r = i >> 6, c = i & 63;
      tc::cp_async16(sm + S::W2 + r * 1024u + ((c ^ (r & 7u)) << 4), q.w2 + (size_t)(rank * S::N2 * 8 + r) * 512 + c * 8, 16u);
    }
    for (int i = tid; i < S::N2 * 8 * 72; i += RT_THREADS) {
      const uint32_t r = i / 72, c = i % 72;
      tc::cp_async16(sm + S::W3 + r * 1152u + ((c ^ (r & 7u)) << 4), q.w3 + (size_t)(rank * S::N2 * 8 + r) * 576 + c * 8, 16u);
    }
    // (the policy's rows of head weights start at multiples of 8 bytes, the value's where the number of actions puts it)
    for (int i = tid; i < A * (S::COLS / 4); i += RT_THREADS) {
      const int k = i / (S::COLS / 4), col = i % (S::COLS / 4) * 4;
      rt_copy_async<8>(sm + S::HEADW + (k * S::COLS + col) * 2, q.wpi + (size_t)k * RT_F + unit_of(col));
    }
    if (tid < S::N1 * 8) rt_copy_async<4>(sm + S::B1 + tid * 4, q.b1 + rank * S::N1 * 8 + tid);
    if (tid < S::N2 * 8) {
      rt_copy_async<4>(sm + S::B2 + tid * 4, q.b2 + rank * S::N2 * 8 + tid);
      rt_copy_async<4>(sm + S::B3 + tid * 4, q.b3 + rank * S::N2 * 8 + tid);
    }
    if (tid < S::COLS) rt_copy_async<4>(sm + S::BFC + tid * 4, q.bfc + unit_of(tid));
    if (tid <= A) rt_copy_async<4>(sm + S::BHEAD + tid * 4, tid < A ? q.bpi + tid : q.bv);
  }
  if (fc)
    for (int i = tid; i < RT_TILE * kbs * 8; i += RT_THREADS) {
      const uint32_t r = i / (kbs * 8), c = i % (kbs * 8);
      tc::cp_async16(sm + S::WFC + r * RT_FC_LD + ((c ^ (r & 7u)) << 4), q.wfc + (size_t)(unit0 + r) * 3136 + kb0 * 64 + c * 8, 16u);
    }
  tc::cp_async_commit();
  if (conv && tid < S::COLS) reinterpret_cast<bf16*>(rt_smem + S::HEADW)[A * S::COLS + tid] = q.wv[unit_of(tid)];
  const uint64_t step0 = *q.step_base + q.t0;
  if (pulls) {
    const size_t at = (size_t)e * STACK_ITEMS + px_lo + tid;
    stack_sixteen(plane, (q.host.fresh[e >> 5] >> (e & 31)) & 1u, reinterpret_cast<const uint4*>(q.host.prev) + 4 * at,
                  reinterpret_cast<uint4*>(const_cast<uint8_t*>(q.frames)) + 4 * at);
  }
  if (q.host.states != nullptr && conv)
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (st_lo + tid + i * RT_THREADS < st_hi) reinterpret_cast<uint4*>(const_cast<uint8_t*>(q.frames))[(size_t)e * (FRAME_WORDS / 4) + st_lo + tid + i * RT_THREADS] = whole[i];
  tc::cp_async_wait<0>();
  __syncthreads();
  rt_cluster_sync();                           // the other blocks have started: their shared memory may be written (and the state is there)
  uint32_t phase = 0u;                         // of the maps' barriers
  // this block's share of a map, complete here, to the others; then wait for theirs
  auto exchange = [&](uint64_t* bar, uint32_t at, uint32_t bytes) {
    tc::fence_proxy_async_smem();
    __syncthreads();
    if (tid == 0) {
      tc::mbar_arrive_expect_tx(bar, (C - 1) * bytes);
#pragma unroll
      for (int c = 1; c < C; ++c) {
        const uint32_t to = (uint32_t)(rank + c) % C;
        rt_send_bulk(rt_map(at, to), at, bytes, rt_map(tc::smem_u32(bar), to));
      }
    }
    if (!s_dead) tc::mbar_wait_limit(bar, phase, &s_dead, q.error_word, tc::ERR_WAIT_FULL, 2u * q.polls);
  };

  for (int t = 0; t < q.steps; ++t) {
    if (t > 0 && __syncthreads_or(s_dead)) break;         // (the last step's frame, and all reads of its rows, are done)
    const uint32_t tag = epoch + 1u + (uint32_t)t;
    const size_t slot = (size_t)t * n;
    // ---- convolutions ----
    if (conv) {
      uint4* frame = reinterpret_cast<uint4*>(rt_smem + S::FRAME);
      if (t == 0) {
        const uint4* src = reinterpret_cast<const uint4*>(q.frames + (size_t)e * FRAME_BYTES);
        for (int i = tid; i < FRAME_WORDS / 4; i += RT_THREADS) frame[i] = __ldcg(src + i);
      } else {
        // the state the last step reached: for this block, and its share for everyone
        const EnvFrame f = s_frame;
        uint8_t* states = t < q.sample_steps ? const_cast<uint8_t*>(q.frames) + (size_t)t * q.frame_step : q.next_frames;
        uint4* out = reinterpret_cast<uint4*>(states + (size_t)e * FRAME_BYTES);
        const int lo = FRAME_WORDS / 4 * rank / C, hi = FRAME_WORDS / 4 * (rank + 1) / C;
#pragma unroll
        for (int k = 0; k < (FRAME_WORDS / 4 + RT_THREADS - 1) / RT_THREADS; ++k) {
          const int i = tid + k * RT_THREADS;
          if (i >= FRAME_WORDS / 4) break;
          const uint4 v = env_frame_quad(f, (uint32_t)i, q.pattern_actions);
          frame[i] = v;
          if (i >= lo && i < hi) out[i] = v;
        }
      }
      __syncthreads();
      if (warp < 13) rt_conv1<C>(rt_smem, sm, q, e, rank, warp, lane);
      exchange(&s_map1, sm + S::ACT1 + rank * S::N1 * RT_PLANE1, S::N1 * RT_PLANE1);
      // The sums of odd tap columns (second layer: the right pixel pair, third layer: the middle column) are taken by other warps
      // than those of even ones and handed over where the frame lay.  One such warp to a scheduler.
      float4* hand = reinterpret_cast<float4*>(rt_smem + S::FRAME) + lane;
      if (warp < 4) {
        const int mg = warp & 1, hi = warp >> 1;
        const uint32_t map1 = sm + S::ACT1 + (lane >> 4) * RT_PLANE1;
        int r0[3];
#pragma unroll
        for (int m = 0; m < 3; ++m) { const int p = min((3 * mg + m) * 16 + (lane & 15), 80); r0[m] = (p / 9) * RT_ROW1 + p % 9 + hi; }
        float acc[3][S::N2][4];
        rt_chain<3, S::N2, 4>(acc, sm + S::W2, 1024, lane, [&](int m, int i, int kk) { return map1 + (kk & 1) * (2 * RT_PLANE1) + (r0[m] + ((i & 1) * 10 + (i >> 1)) * RT_ROW1 + 10 * (kk >> 1)) * 16; },
                              [&](int i) { return 2 * i + hi; });
        if (hi) {
#pragma unroll
          for (int m = 0; m < 3; ++m)
#pragma unroll
            for (int j = 0; j < S::N2; ++j) hand[((3 * mg + m) * S::N2 + j) * 32] = make_float4(acc[m][j][0], acc[m][j][1], acc[m][j][2], acc[m][j][3]);
        }
        rt_pair_sync(1 + mg);
        if (!hi) {
#pragma unroll
          for (int j = 0; j < S::N2; ++j) {
            const int nt = rank * S::N2 + j;
            const float2 b = *reinterpret_cast<const float2*>(rt_smem + S::B2 + (j * 8 + 2 * t4) * 4);
#pragma unroll
            for (int m = 0; m < 3; ++m) {
              const float4 o = hand[((3 * mg + m) * S::N2 + j) * 32];
              const uint32_t v[2] = {rt_relu_pack((o.x + acc[m][j][0]) + b.x, (o.y + acc[m][j][1]) + b.y),
                                     rt_relu_pack((o.z + acc[m][j][2]) + b.x, (o.w + acc[m][j][3]) + b.y)};
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                const int p = (3 * mg + m) * 16 + g + 8 * i;
                if (p < 81) rt_sts(sm + S::ACT2 + nt * RT_PLANE2 + (p / 9 * RT_ROW2 + p % 9) * 16 + 4 * t4, v[i]);
              }
            }
          }
        }
      } else {
        // the other warps write the block's share of the first layer's map out
        uint4* out = reinterpret_cast<uint4*>(q.act1 + (slot + e) * TC1::OUT_SIZE);
        for (int i = 1600 * rank / C + tid - 128; i < 1600 * (rank + 1) / C; i += RT_THREADS - 128) {
          const int c = i & 3, y = i / 80, x = (i >> 2) - 20 * y;
          out[i] = *reinterpret_cast<const uint4*>(rt_smem + S::ACT1 + c * RT_PLANE1 + rt_place1(y, x) * 16);
        }
      }
      exchange(&s_map2, sm + S::ACT2 + rank * S::N2 * RT_PLANE2, S::N2 * RT_PLANE2);
      phase ^= 1u;
      if (warp < 4) {
        const int mg = warp & 1, hi = warp >> 1;
        const uint32_t map2 = sm + S::ACT2 + (lane >> 4) * RT_PLANE2;
        int r0[2];
#pragma unroll
        for (int m = 0; m < 2; ++m) { const int p = min((2 * mg + m) * 16 + (lane & 15), RT_POS3 - 1); r0[m] = (p / 7) * RT_ROW2 + p % 7; }
        float acc[2][S::N2][4];
        if (hi) rt_chain<2, S::N2, 3>(acc, sm + S::W3, 1152, lane, [&](int m, int i, int kk) { return map2 + kk * (2 * RT_PLANE2) + (r0[m] + RT_ROW2 * i + 1) * 16; },
                                      [](int i) { return 3 * i + 1; });
        else rt_chain<2, S::N2, 6>(acc, sm + S::W3, 1152, lane, [&](int m, int i, int kk) { return map2 + kk * (2 * RT_PLANE2) + (r0[m] + RT_ROW2 * (i >> 1) + 2 * (i & 1)) * 16; },
                                   [](int i) { return 3 * (i >> 1) + 2 * (i & 1); });
        if (hi) {
#pragma unroll
          for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int j = 0; j < S::N2; ++j) hand[((2 * mg + m) * S::N2 + j) * 32] = make_float4(acc[m][j][0], acc[m][j][1], acc[m][j][2], acc[m][j][3]);
        }
        rt_pair_sync(1 + mg);
        if (!hi) {
#pragma unroll
          for (int j = 0; j < S::N2; ++j) {
            const int ch = (rank * S::N2 + j) * 8 + 2 * t4;
            const float2 b = *reinterpret_cast<const float2*>(rt_smem + S::B3 + (j * 8 + 2 * t4) * 4);
#pragma unroll
            for (int m = 0; m < 2; ++m) {
              const float4 o = hand[((2 * mg + m) * S::N2 + j) * 32];
              const uint32_t v[2] = {rt_relu_pack((o.x + acc[m][j][0]) + b.x, (o.y + acc[m][j][1]) + b.y),
                                     rt_relu_pack((o.z + acc[m][j][2]) + b.x, (o.w + acc[m][j][3]) + b.y)};
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                const int p = (2 * mg + m) * 16 + g + 8 * i;
                if (p >= RT_POS3) continue;
                word_store(reinterpret_cast<uint2*>(q.maps) + ((size_t)e * RT_POS3 + p) * 32 + ch / 2, v[i], tag);
                *reinterpret_cast<uint32_t*>(q.act3 + (slot + e) * TC3::OUT_SIZE + p * 64 + ch) = v[i];
              }
            }
          }
        }
      } else {
        uint4* out = reinterpret_cast<uint4*>(q.act2 + (slot + e) * TC2::OUT_SIZE);
        for (int i = 648 * rank / C + tid - 128; i < 648 * (rank + 1) / C; i += RT_THREADS - 128) {
          out[i] = *reinterpret_cast<const uint4*>(rt_smem + S::ACT2 + (i & 7) * RT_PLANE2 + ((i >> 3) / 9 * RT_ROW2 + (i >> 3) % 9) * 16);
        }
      }
      __syncthreads();
    }
    // ---- fully connected layer: this block's slice of K and units, for all states ----
    if (fc)
      for (int row0 = 0; row0 < n; row0 += RT_ROWS) {
        const int rows = min(RT_ROWS, n - row0);
        const uint32_t u = tid & 15;
        for (int r = tid >> 4; r < rows; r += RT_THREADS / 16) {
          const uint4* src = q.maps + ((size_t)(row0 + r) * RT_POS3 + kb0) * 16 + u;
          uint4 v[7];
          word_await(v, src, 16, kbs, tag, &s_dead, q.error_word, q.polls);
#pragma unroll
          for (int p = 0; p < 7; ++p)
            if (p < kbs) {
              *reinterpret_cast<uint2*>(rt_smem + S::ROWS + r * RT_FC_LD + (((uint32_t)(p * 8 + (u >> 1)) ^ (r & 7u)) << 4) + (u & 1) * 8) = make_uint2(v[p].x, v[p].z);
            }
        }
        __syncthreads();
        const int mt = warp >> 1, np = warp & 1;                       // sixteen states, sixteen units
        if (mt * 16 < rows) {
          float acc[2][4] = {};
          const uint32_t ar = (uint32_t)(mt * 16 + (lane & 15)), br = (uint32_t)(np * 16 + (lane & 7) + (lane >> 4) * 8);
          const uint32_t ab = sm + S::ROWS + ar * RT_FC_LD, bb = sm + S::WFC + br * RT_FC_LD, ah = (uint32_t)lane >> 4, bh = ((uint32_t)lane >> 3) & 1u;
          uint32_t a[2][4][4], b[2][4][4];
          auto load = [&](int kb, int into) {                         // 64 k: pieces of eight
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              rt_ldsm4(ab + kb * 128 + ((2u * i + ah) ^ (ar & 7u)) * 16u, a[into][i]);
              rt_ldsm4(bb + kb * 128 + ((2u * i + bh) ^ (br & 7u)) * 16u, b[into][i]);
            }
          };
          load(0, 0);
#pragma unroll
          for (int kb = 0; kb < 7; ++kb) {
            if (kb + 1 < kbs) load(kb + 1, (kb + 1) & 1);
            if (kb < kbs)
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                rt_mma_bf16(acc[0], a[kb & 1][i], b[kb & 1][i][0], b[kb & 1][i][1]);
                rt_mma_bf16(acc[1], a[kb & 1][i], b[kb & 1][i][2], b[kb & 1][i][3]);
              }
          }
#pragma unroll
          for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const int r = row0 + mt * 16 + g + 8 * i;
              if (r < n)
                word_store(q.sums + ((size_t)slice * n + r) * 256 + (unit0 + np * 16 + j * 8 + 2 * t4) / 2, __float_as_uint(acc[j][2 * i]),
                           __float_as_uint(acc[j][2 * i + 1]), tag);
            }
        }
        __syncthreads();
      }
    if (!conv) continue;
    // ---- the end of the state's pass: this block's hidden units and their part of the heads ----
    const bool sample = t < q.sample_steps, stepping = sample && q.env;
    if (stepping && lane == 0 && warp == 8) s_prep = env_prepare(q.seed, (uint32_t)e, n, (uint32_t)step0 + t, rank == 0 ? q.counters : nullptr);
    float* xs = reinterpret_cast<float*>(rt_smem + S::XS);
    if (tid < S::COLS / 2) {
      const int col = tid * 2, u = unit_of(col);
      const uint4* src = q.sums + (size_t)e * 256 + u / 2;
      uint4 v[RT_SLICES];
      word_await(v, src, (size_t)n * 256, RT_SLICES, tag, &s_dead, q.error_word, q.polls);
      float s0 = 0.f, s1 = 0.f;
#pragma unroll
      for (int s = 0; s < RT_SLICES; ++s) {
        s0 += __uint_as_float(v[s].x); s1 += __uint_as_float(v[s].z);
      }
      const float2 b = *reinterpret_cast<const float2*>(rt_smem + S::BFC + col * 4);
      const __nv_bfloat162 x = __floats2bfloat162_rn(fmaxf(s0 + b.x, 0.f), fmaxf(s1 + b.y, 0.f));
      *reinterpret_cast<__nv_bfloat162*>(q.h + (slot + e) * RT_F + u) = x;
      *reinterpret_cast<float2*>(xs + col) = __bfloat1622float2(x);
    }
    __syncthreads();
    {
      // RUNS lanes to a head output: each its running sum over four groups of four units, then the tree over this block's sums
      constexpr int PER = 32 / S::RUNS;
      const int run = lane % S::RUNS, outputs = A + 1;
      for (int o0 = warp * PER; o0 < outputs; o0 += RT_WARPS * PER) {
        const int k = min(o0 + lane / S::RUNS, outputs - 1);
        float acc0 = 0.f, acc1 = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float4 x = *reinterpret_cast<const float4*>(xs + 4 * (run + S::RUNS * j));
          const uint2 w = *reinterpret_cast<const uint2*>(rt_smem + S::HEADW + (k * S::COLS + 4 * (run + S::RUNS * j)) * 2);
          acc0 = fmaf(__uint_as_float(w.x << 16), x.x, acc0);
          acc1 = fmaf(__uint_as_float(w.x & 0xFFFF0000u), x.y, acc1);
          acc0 = fmaf(__uint_as_float(w.y << 16), x.z, acc0);
          acc1 = fmaf(__uint_as_float(w.y & 0xFFFF0000u), x.w, acc1);
        }
        float v = acc0 + acc1;
#pragma unroll
        for (int b = S::RUNS / 2; b > 0; b >>= 1) v += __shfl_xor_sync(0xffffffffu, v, b);
        if (run < C && o0 + lane / S::RUNS < outputs)
          rt_send(rt_map(sm + S::ZS + (uint32_t)(rank * 36 + k) * 4u, run), __float_as_uint(v), rt_map(tc::smem_u32(&s_heads), run));
      }
      if (tid == 0) tc::mbar_arrive_expect_tx(&s_heads, (uint32_t)(C * outputs * 4));
    }
    if (warp == 0 && !s_dead) tc::mbar_wait_limit(&s_heads, t & 1, &s_dead, q.error_word, tc::ERR_WAIT_FULL, 2u * q.polls);
    if (warp == 0) {
      const float* z = reinterpret_cast<const float*>(rt_smem + S::ZS);
      float s = -INFINITY;
      if (lane <= A) {
        if constexpr (C == 2) s = z[lane] + z[36 + lane];
        else s = (z[lane] + z[36 + lane]) + (z[72 + lane] + z[108 + lane]);
        s += reinterpret_cast<const float*>(rt_smem + S::BHEAD)[lane];
      }
      const int32_t a = warp_finish_heads(q.mode, lane < A ? s : -INFINITY, __shfl_sync(0xffffffffu, s, A), lane, A, (size_t)e, q.logits + slot * A,
                                          q.values + slot, sample, q.seed, step0 + t, q.forced ? q.forced + slot : nullptr, q.actions + slot,
                                          q.sampled + slot, q.uniforms + slot);
      if (q.host.done != nullptr && rank == 0 && lane == 0) {
        if (sample) q.host.actions[e] = a;
        q.host.values[e] = q.values[slot + e];
        __threadfence_system();
      }
      if (stepping && lane == 0) {
        const EnvPrep prep = s_prep;
        const EnvOutcome o = env_outcome(prep, a, q.term_denom, q.pattern_actions);
        s_frame = env_frame_of(prep.pre_next, o.tag, q.pattern_actions);
        if (rank == 0) env_record(prep, o, (uint32_t)e, n, q.rewards + slot, q.terminals + slot, q.counters);
      }
    }
  }
  // Nobody leaves before all that others send it has arrived: it waited for that, unless it gave up.  Then, once every block of the cluster
  // has sent its last, all of them stay for 100 us (a copy takes about one).
  if (__syncthreads_or(s_dead) && tid < C) rt_store(rt_map(tc::smem_u32(const_cast<uint32_t*>(&s_linger)), tid), 1u);
  rt_cluster_sync();
  if (s_linger) {
    for (int i = 0; i < 100; ++i) __nanosleep(1000u);
    rt_cluster_sync();
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

template <int C_> struct RtKernel {
  static constexpr int C = C_;
  static auto kernel() { return rollout_tc_kernel<C>; }
  static void shape(cudaLaunchConfig_t& cfg, cudaLaunchAttribute& attr, int clusters) {
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3(clusters * C); cfg.blockDim = dim3(RT_THREADS); cfg.dynamicSmemBytes = RtMem<C>::TOTAL;
    attr.id = cudaLaunchAttributeCooperative; attr.val.cooperative = 1;
    cfg.attrs = &attr; cfg.numAttrs = 1;
  }
  // Clusters that are resident at once (blocks that wait for one another have to be); 0 if they are too few for the fully
  // connected layer's tiles.
  static int clusters() {
    static const int most = [] {
      cudaLaunchConfig_t cfg;
      cudaLaunchAttribute attr;
      shape(cfg, attr, 1);
      cfg.numAttrs = 0;
      int dev = 0, coop = 0, count = 0;
      const bool known = cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess &&
                         cudaFuncSetAttribute(kernel(), cudaFuncAttributeMaxDynamicSharedMemorySize, RtMem<C>::TOTAL) == cudaSuccess &&
                         cudaOccupancyMaxActiveClusters(&count, kernel(), &cfg) == cudaSuccess;
      if (!known) cudaGetLastError();
      return known && coop != 0 && count * C >= RT_FC_BLOCKS ? count : 0;
    }();
    return most;
  }
};
template <class F> static auto rt_pick(int n, F f) {
  if (n <= RtKernel<4>::clusters()) return f(RtKernel<4>{});
  return f(RtKernel<2>{});
}

// One environment per cluster: up to there the launches this replaces take 115 to 130 us a rollout (five steps and the bootstrap pass)
// and this kernel 66 to 92.  With a second environment for some clusters it takes 135 us at 75 and 154 at 148, against 130 and 157.
constexpr int RT_MOST = 74;
bool rollout_tc_supported(int n, int n_actions) {
  return n <= RT_MOST && n_actions < 32 && tc_fc_slices(n) == RT_SLICES && rt_pick(n, [&](auto k) { return n <= k.clusters(); });
}
static size_t rt_map_words(int n) { return (size_t)n * RT_POS3 * 16; }
size_t rollout_tc_words(int n) { return n > RT_MOST ? 0 : rt_map_words(n) + (size_t)n * RT_SLICES * 256; }

void launch_rollout_tc(LaunchCtx& lc, const NetDims& nd, const float* theta, const bf16* theta16, const bf16* images, const SmallRollout& r) {
  const LayerDims* d = nd.layer;
  RtArgs q{};
  q.n = r.n; q.A = nd.A; q.steps = r.steps; q.t0 = r.t0;
  q.frames = r.frames; q.frame_step = r.frame_step; q.next_frames = r.env.next_frames; q.sample_steps = r.sample_steps; q.env = r.step_env;
  q.w1 = (const __half*)tc_conv1_weights(images); q.w2 = theta16 + d[1].w_off; q.w3 = theta16 + d[2].w_off; q.wfc = theta16 + d[3].w_off; q.wpi = theta16 + nd.pi_w;
  q.wv = theta16 + nd.v_w; q.b1 = theta + d[0].b_off; q.b2 = theta + d[1].b_off; q.b3 = theta + d[2].b_off; q.bfc = theta + d[3].b_off;
  q.bpi = theta + nd.pi_b; q.bv = theta + nd.v_b; q.scale1 = tc_conv1_scale();
  q.act1 = (bf16*)r.act[0]; q.act2 = (bf16*)r.act[1]; q.act3 = (bf16*)r.act[2]; q.h = (bf16*)r.act[3];
  q.maps = (uint4*)r.words; q.sums = q.maps + rt_map_words(r.n); q.sync = r.sync;
  q.logits = r.logits; q.values = r.values; q.uniforms = r.uniforms; q.actions = r.actions; q.sampled = r.sampled; q.counters = r.env.counters;
  q.forced = r.forced; q.rewards = r.env.rewards; q.terminals = r.env.terminals; q.seed = r.seed; q.step_base = r.step_base; q.advance = r.advance;
  q.term_denom = r.env.term_denom; q.pattern_actions = r.env.pattern_actions; q.mode = r.mode; q.host = r.host; q.error_word = r.error_word;
  q.polls = r.polls;
  lc.serialize_next = false;
  KernelScope scope(lc, KID_SMALL_ROLLOUT);
  const bool launched = rt_pick(r.n, [&](auto k) {
    typedef decltype(k) Kernel;
    const int clusters = Kernel::clusters();
    if (clusters == 0) return false;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr;
    Kernel::shape(cfg, attr, clusters);
    cfg.stream = lc.st;
    return cudaLaunchKernelEx(&cfg, Kernel::kernel(), q) == cudaSuccess;
  });
  if (!launched) lc.host_failure = true;
}

}  // namespace paac
