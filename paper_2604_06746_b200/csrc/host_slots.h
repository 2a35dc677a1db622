// Words in mapped host memory that the device writes for the host, each below the tag of the call it belongs to: a slot of them
// per context, shared out by one table per process.  No CUDA here (api.cu allocates the memory and asks about the stream).
#pragma once

#include <cstring>

namespace skv {

constexpr int kSlots = 64, kSlotWords = 144;

struct HostSlot {
  unsigned long long* mem;               // [kSlotWords], mapped
  unsigned seq;                          // tag of the last call; it goes on from owner to owner, so that no word is taken for another's
  bool used;
  bool awaited;                          // words of the last call may still be on their way
};

// A free slot, or NULL.  `mem` holds zeros at first.
inline HostSlot* take_slot(HostSlot (&slots)[kSlots], unsigned long long* mem) {
  for (int i = 0; i < kSlots; ++i)
    if (!slots[i].used) {
      slots[i].used = true;
      slots[i].mem = mem + i * kSlotWords;
      return &slots[i];
    }
  return nullptr;
}
// A slot whose words were not all seen (a call that failed) stays out: they could come over those of its next owner.
inline void give_back_slot(HostSlot* s) { s->used = s->awaited; }

// The tag of the next call, never that of clean words.
inline unsigned next_tag(HostSlot& s) {
  s.awaited = true;
  if (++s.seq == 0) ++s.seq;
  return s.seq;
}

// Waits for the last call's words: the pivot and one of each layer, those that nobody asked for too, so that none is on its way
// once this returns.  done() (asked now and then): 0 while the stream works, 1 once it is through, -1 after an error.
template <class F>
bool await_words(HostSlot& s, int n_layers, int* pivot_out, float* t_out, F done) {
  const volatile unsigned long long* mem = s.mem;
  unsigned spins = 0;
  for (int i = 0; i <= n_layers; ++i) {
    unsigned long long word;
    while ((unsigned)((word = mem[i]) >> 32) != s.seq) {
      if (++spins % 100000 != 0) continue;               // tens of microseconds
      const int state = done();
      if (state == 0) continue;
      if (state < 0 || (unsigned)(mem[i] >> 32) != s.seq) return false;   // through, and no word
    }
    const unsigned value = (unsigned)word;
    if (i == 0) *pivot_out = (int)value;
    else if (t_out) std::memcpy(&t_out[i - 1], &value, sizeof(float));
  }
  s.awaited = false;
  return true;
}

}  // namespace skv
