// The synthetic environments' transition and frame, shared by the kernels that step them (one block per environment).
#pragma once
#include "common.cuh"

namespace paac {

constexpr int FRAME_WORDS = FRAME_H * FRAME_W;   // 7056, a multiple of 4

// What of a transition does not depend on the action: prepared by one thread while the action is being found.  Without `counters` (a
// block that will not record the transition, beside one that may be writing them) those are left out.
struct EnvPrep { uint32_t pre_step, pre_next; int32_t len, ret, episodes; };
__device__ __forceinline__ EnvPrep env_prepare(uint64_t seed, uint32_t e, int n_e, uint32_t step, const int32_t* counters) {
  EnvPrep p;
  p.pre_step = env_hash_prefix(seed, e, step);
  p.pre_next = env_hash_prefix(seed, e, step + 1u);
  p.len = p.ret = p.episodes = 0;
  if (counters != nullptr) { p.len = counters[e]; p.ret = counters[n_e + e]; p.episodes = counters[2 * n_e + e]; }
  return p;
}
// the frame of a state: its hash base, and the band of the learnable environment in pixel words (empty otherwise)
struct EnvFrame { uint32_t base, band_lo, band_hi; };
// pattern_actions > 0: the learnable environment.  The state at step k of environment e has the goal
// hash(e, k, 'GOAL') mod A; its frame is the hashed frame with every byte reduced to its low six bits (a dim
// texture) and rows [band goal, band (goal + 1)), band = 84 / A, set to 255; an action pays 1 if it is the current
// state's goal and 0 otherwise.
__device__ __forceinline__ EnvFrame env_frame_of(uint32_t pre_next, uint32_t tag, int pattern_actions) {
  EnvFrame f{hash_mix(pre_next ^ tag), 0u, 0u};
  if (pattern_actions > 0) {
    const uint32_t goal = hash_mix(hash_mix(pre_next) ^ HASH_TAG_GOAL) % (uint32_t)pattern_actions;
    const uint32_t band = (uint32_t)(FRAME_H / pattern_actions);
    f.band_lo = band * goal * FRAME_W;                  // a row is 84 words, so four words never straddle it
    f.band_hi = f.band_lo + band * FRAME_W;
  }
  return f;
}
struct EnvOutcome { int reward; bool terminal; uint32_t tag; };
__device__ __forceinline__ EnvOutcome env_outcome(const EnvPrep& p, int32_t a, uint32_t term_denom, int pattern_actions) {
  EnvOutcome o;
  const uint32_t base = hash_mix(p.pre_step ^ ((uint32_t)a + 1u));
  const uint32_t hr = hash_mix(base ^ HASH_TAG_REWARD) & 15u;
  o.reward = hr == 0u ? 1 : (hr == 1u ? -1 : 0);
  if (pattern_actions > 0)
    o.reward = (uint32_t)a == hash_mix(hash_mix(p.pre_step) ^ HASH_TAG_GOAL) % (uint32_t)pattern_actions ? 1 : 0;
  const uint32_t hterm = hash_mix(base ^ HASH_TAG_TERMINAL);
  o.terminal = (uint32_t)(((uint64_t)hterm * term_denom) >> 32) == 0u;
  o.tag = o.terminal ? 0u : (uint32_t)a + 1u;
  return o;
}
__device__ __forceinline__ void env_record(const EnvPrep& p, const EnvOutcome& o, uint32_t e, int n_e, int8_t* rewards,
                                           uint8_t* terminals, int32_t* counters) {
  rewards[e] = (int8_t)o.reward;
  terminals[e] = o.terminal ? 1 : 0;
  if (o.terminal) counters[2 * n_e + e] = p.episodes + 1;
  counters[e] = o.terminal ? 0 : p.len + 1;
  counters[n_e + e] = o.terminal ? 0 : p.ret + o.reward;
}
// sixteen bytes of a frame: one hashed 32-bit word per pixel (its bytes, little endian, are the four channels)
__device__ __forceinline__ uint4 env_frame_quad(const EnvFrame f, uint32_t q, int pattern_actions) {
  const uint32_t keep = pattern_actions > 0 ? 0x3F3F3F3Fu : 0xFFFFFFFFu, p = q * 4u + 1u;
  if (q * 4u >= f.band_lo && q * 4u < f.band_hi) return make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu);
  return make_uint4(hash_mix(f.base + HASH_K0 * p) & keep, hash_mix(f.base + HASH_K0 * (p + 1u)) & keep,
                    hash_mix(f.base + HASH_K0 * (p + 2u)) & keep, hash_mix(f.base + HASH_K0 * (p + 3u)) & keep);
}
// the whole block writes the 84 x 84 x 4 frame
template <int THREADS>
__device__ __forceinline__ void env_write_frame(const EnvFrame f, uint8_t* frame, int pattern_actions) {
  uint4* out = reinterpret_cast<uint4*>(frame);
  for (int q = threadIdx.x; q < FRAME_WORDS / 4; q += THREADS) out[q] = env_frame_quad(f, (uint32_t)q, pattern_actions);
}

// Sixteen pixels of a frame stack: out = (three newest channels of prev, the plane's pixel), or four copies of the pixel for a fresh one.
constexpr int STACK_ITEMS = FRAME_H * FRAME_W / 16;
static_assert(STACK_ITEMS * 16 == FRAME_H * FRAME_W, "whole 16-byte words");
__device__ __forceinline__ void stack_sixteen(const uint4 plane, bool fresh, const uint4* prev, uint4* out) {
  const uint32_t w[4] = {plane.x, plane.y, plane.z, plane.w};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    uint4 o;
    if (fresh) {
      o = make_uint4((w[q] & 0xFFu) * 0x01010101u, ((w[q] >> 8) & 0xFFu) * 0x01010101u, ((w[q] >> 16) & 0xFFu) * 0x01010101u, (w[q] >> 24) * 0x01010101u);
    } else {
      const uint4 p = prev[q];
      o = make_uint4((p.x >> 8) | (w[q] << 24), (p.y >> 8) | ((w[q] >> 8) << 24), (p.z >> 8) | ((w[q] >> 16) << 24), (p.w >> 8) | ((w[q] >> 24) << 24));
    }
    out[q] = o;
  }
}

}  // namespace paac
