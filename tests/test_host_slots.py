"""Slots of host words (csrc/host_slots.h), on the CPU: a small program compiled against the header.  What one owner's call leaves
late must neither pass for the next owner's words nor come over them."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_06746_b200", "csrc")
MAIN = r"""
#include <cstdio>
#include <cstring>
#include "host_slots.h"
using namespace skv;
static HostSlot slots[kSlots];
static unsigned long long mem[kSlots * kSlotWords];
static unsigned long long word(unsigned tag, unsigned v) { return (unsigned long long)tag << 32 | v; }
#define CHECK(x) if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; }

int main() {
  int pivot = -1;
  // the pivot's word first, the layers' while the host waits: a call without t_out returns after those too
  HostSlot* a = take_slot(slots, mem);
  unsigned tag = next_tag(*a);
  a->mem[0] = word(tag, 3);
  int asked = 0;
  auto late = [&]() {
    ++asked;
    for (int l = 0; l < 5; ++l) a->mem[1 + l] = word(tag, 0x3f800000u + l);
    return 0;
  };
  CHECK(await_words(*a, 5, &pivot, nullptr, late) && pivot == 3 && asked == 1);
  // with t_out
  float t[5];
  tag = next_tag(*a);
  a->mem[0] = word(tag, 4);
  CHECK(await_words(*a, 5, &pivot, t, late) && pivot == 4 && t[0] == 1.f && asked == 2);
  // the next owner's tags are others
  give_back_slot(a);
  HostSlot* b = take_slot(slots, mem);
  CHECK(b == a && next_tag(*b) > tag);
  // its stream is through, and the words are not its own: an error, and the slot stays out
  CHECK(!await_words(*b, 5, &pivot, t, []() { return 1; }));
  CHECK(!await_words(*b, 5, &pivot, t, []() { return -1; }));
  give_back_slot(b);
  HostSlot* c = take_slot(slots, mem);
  CHECK(c != b && c->mem == mem + kSlotWords);
  // a slot that nobody used comes back; all of them are there, once
  give_back_slot(c);
  int n = 0;
  while (HostSlot* s = take_slot(slots, mem)) { CHECK(s->mem + kSlotWords <= mem + kSlots * kSlotWords); ++n; }
  CHECK(n == kSlots - 1);
  // tags pass over that of clean words
  c->seq = 0xffffffffu;
  CHECK(next_tag(*c) == 1u);
  return 0;
}
"""


def test_slots(tmp_path):
    src, exe = tmp_path / "main.cpp", tmp_path / "main"
    src.write_text(MAIN)
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
