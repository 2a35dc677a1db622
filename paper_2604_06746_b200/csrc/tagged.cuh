// Words that CTAs of one launch exchange through global memory.  The words of a context start from zero, and every
// launch uses tags that are larger than those before it: whoever sees the tag it waits for sees the value with
// it, in one trip, without fences, flags or anything to clear.
#pragma once

#include "common.cuh"

namespace skv {

// A value and the tag that says whose it is, in one 64-bit word: whoever sees the tag sees the value.
__device__ __forceinline__ unsigned long long tagged(float v, unsigned tag) {
  return (unsigned long long)tag << 32 | __float_as_uint(v);
}
__device__ __forceinline__ float word_value(unsigned long long w) { return __uint_as_float((unsigned)w); }
__device__ __forceinline__ bool word_has(unsigned long long w, unsigned tag) { return (unsigned)(w >> 32) == tag; }
__device__ __forceinline__ void put_word(unsigned long long* p, unsigned long long w) {
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}
__device__ __forceinline__ unsigned long long get_word(const unsigned long long* p) {
  unsigned long long w;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
  return w;
}
// The same for a value that says that others are ready.
__device__ __forceinline__ unsigned long long get_word_acquire(const unsigned long long* p) {
  unsigned long long w;
  asm volatile("ld.acquire.gpu.global.b64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
  return w;
}
// What the last CTA of a launch does, `threads` of its threads: the tags move on to `next`, or, long before they wrap, start
// over with clean words.
__device__ __forceinline__ void pass_tags_on(unsigned long long* xch, int* ctl, unsigned next, int thread, int threads) {
  const bool over = next > 0x7f000000u;
  if (over)
    for (size_t i = thread; i < (size_t)kXchWords; i += threads) xch[i] = 0;
  if (thread == 0) {
    ctl[kCtlTag] = over ? 0 : (int)next;
    ctl[kCtlExit] = 0;
  }
}

}  // namespace skv
