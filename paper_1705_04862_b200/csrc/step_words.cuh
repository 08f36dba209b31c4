// Words that carry the number of the step they belong to beside their value: how the blocks of the one-launch rollouts hand each
// other numbers through L2.  A reader polls the words themselves, so there is neither a barrier (1.2 us over the device) nor a round
// trip for the numbers after it.  Every 8-byte half of an access is (value, step), written and read as one.  A word may be
// overwritten for the next step once all that read it have: the kernels say why that holds.  The step numbers go on from launch
// to launch; the block that ends last moves the count on (sync[0] steps so far, sync[1] blocks that have ended).
//
// Every wait is bounded.  A thread that gives up raises the error word and *dead, with which its block goes on without waiting.
#pragma once
#include "common.cuh"
#include "tc_common.cuh"

namespace paac {

constexpr uint32_t WORD_POLLS = 2000000u;

__device__ __forceinline__ void word_peek(const uint4* p, uint4& v) {
  asm volatile("ld.volatile.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
}
__device__ __forceinline__ void word_peek(const uint2* p, uint2& v) {
  asm volatile("ld.volatile.global.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
}
__device__ __forceinline__ bool word_of(const uint4 v, uint32_t step) { return v.y == step && v.w == step; }
__device__ __forceinline__ bool word_of(const uint2 v, uint32_t step) { return v.y == step; }
__device__ __forceinline__ void word_store(uint4* p, uint32_t a, uint32_t b, uint32_t step) {
  asm volatile("st.volatile.global.v4.u32 [%0], {%1, %2, %3, %2};" ::"l"(p), "r"(a), "r"(step), "r"(b) : "memory");
}
__device__ __forceinline__ void word_store(uint2* p, uint32_t a, uint32_t step) {
  asm volatile("st.volatile.global.v2.u32 [%0], {%1, %2};" ::"l"(p), "r"(a), "r"(step) : "memory");
}
// v[i] = the word at p + i * stride, i < count (of N), once all are of the step, or as they are after a bounded wait.  All are asked
// for together, again and again: one after the other each would cost a round trip through L2.
template <int N, class W>
__device__ __forceinline__ void word_await(W (&v)[N], const W* p, size_t stride, int count, uint32_t step, volatile uint32_t* dead, uint32_t* error_word) {
  for (uint32_t polls = 0;; ++polls) {
    bool ready = true;
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (i < count) word_peek(p + i * stride, v[i]);
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (i < count) ready = ready && word_of(v[i], step);
    if (ready || *dead) return;
    if (polls == WORD_POLLS) { *dead = 1u; atomicOr(error_word, tc::ERR_WAIT_FULL); return; }
  }
}

}  // namespace paac
