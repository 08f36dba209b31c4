// Words that carry the number of the step they belong to beside their value: how the blocks of the one-launch rollouts hand each
// other numbers through L2 (a flag in the same store as the data, as collective libraries send short messages).  A reader polls the
// words themselves, so there is neither a barrier (1.2 us over the device) nor a round trip for the numbers after it.  Every 8-byte
// half of an access is (value, step) packed into one 64-bit element, as the memory model keeps an element whole but takes a vector's
// elements one by one, in any order: of two 32-bit elements a reader might see the new step beside the old value.  A word may be
// overwritten for the next step once all that read it have: the kernels say why that holds.  The step numbers go on from launch
// to launch; the block that ends last moves the count on (sync[0] steps so far, sync[1] blocks that have ended).
//
// Every wait is bounded (`limit` polls; WORD_POLLS, of the order of a second, unless a test asks for less).  A thread that gives up
// raises the error word and *dead, with which its block goes on without waiting.
#pragma once
#include "common.cuh"
#include "tc_common.cuh"

namespace paac {

__device__ __forceinline__ uint64_t word_half(uint32_t value, uint32_t step) { return (uint64_t)step << 32 | value; }
__device__ __forceinline__ void word_peek(const uint4* p, uint4& v) {
  uint64_t a, b;
  asm volatile("ld.volatile.global.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
  v = make_uint4((uint32_t)a, (uint32_t)(a >> 32), (uint32_t)b, (uint32_t)(b >> 32));
}
__device__ __forceinline__ void word_peek(const uint2* p, uint2& v) {
  uint64_t a;
  asm volatile("ld.volatile.global.b64 %0, [%1];" : "=l"(a) : "l"(p) : "memory");
  v = make_uint2((uint32_t)a, (uint32_t)(a >> 32));
}
__device__ __forceinline__ bool word_of(const uint4 v, uint32_t step) { return v.y == step && v.w == step; }
__device__ __forceinline__ bool word_of(const uint2 v, uint32_t step) { return v.y == step; }
__device__ __forceinline__ void word_store(uint4* p, uint32_t a, uint32_t b, uint32_t step) {
  asm volatile("st.volatile.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(word_half(a, step)), "l"(word_half(b, step)) : "memory");
}
__device__ __forceinline__ void word_store(uint2* p, uint32_t a, uint32_t step) {
  asm volatile("st.volatile.global.b64 [%0], %1;" ::"l"(p), "l"(word_half(a, step)) : "memory");
}
// v[i] = the word at p + i * stride, i < count (of N), once all are of the step, or as they are after a bounded wait.  All are asked
// for together, again and again: one after the other each would cost a round trip through L2.
template <int N, class W>
__device__ __forceinline__ void word_await(W (&v)[N], const W* p, size_t stride, int count, uint32_t step, volatile uint32_t* dead, uint32_t* error_word,
                                           uint32_t limit) {
  for (uint32_t polls = 0;; ++polls) {
    bool ready = true;
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (i < count) word_peek(p + i * stride, v[i]);
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (i < count) ready = ready && word_of(v[i], step);
    if (ready || *dead) return;
    if (polls == limit) { *dead = 1u; atomicOr(error_word, tc::ERR_WAIT_FULL); return; }
  }
}

}  // namespace paac
