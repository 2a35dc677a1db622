// Rank search over fp32 keys held in registers (token selection).  A cluster of CL CTAs of kRxThreads threads
// shares one vector; digits of 11, 11 and 10 bits from the top.  Each level: keys are counted into a histogram of
// 2048 bins (four copies of a bin, one for every fourth lane); 32 warps add up 64 bins each, the 32 sums go to every CTA
// of the cluster, and one warp walks them and then the 64 bins that hold the wanted rank (all 32 of them: 1760
// clocks a level in one CTA instead of 1350, and 131072 keys in a cluster 103 us).  In a cluster the bins come through
// distributed shared memory, already summed over their copies.
// Three block barriers a level; one pass over memory in all where the vector fits the registers.
// Bound by the chain of barriers and shared-memory round trips.  us for 1777 / 8192 / 32768 / 131072 keys: 5.1 / 7.2 / 9.4 /
// 18.7 with the copies read by every walker and a branch around each count, now 4.5 / 5.1 / 6.6 / 12.5; four levels of eight
// bits with a copy of every bin per lane took 7.5 us for 1000 keys and 22.3 for 131072.
#pragma once

#include <cooperative_groups.h>

#include "common.cuh"

namespace skv {

namespace cg = cooperative_groups;

constexpr int kRxThreads = 1024;
constexpr int kRxLevels = 3, kRxBins = 2048, kRxCopies = 4;

template <int CL>
struct RadixShared {
  uint4 hist[kRxLevels][kRxBins];      // copies of a bin
  unsigned bins[kRxLevels][CL > 1 ? kRxBins : 1];      // clusters: their sums, which the others read
  unsigned sums[kRxLevels][CL][32];    // of 64 bins each, of every CTA of the cluster
  unsigned found[kRxLevels][3];        // digit, keys in it, rank in it
  unsigned scratch[2][32];             // counts of the warps
};
__device__ __forceinline__ int radix_shift(int level) { return level == 0 ? 21 : level == 1 ? 10 : 0; }
__device__ __forceinline__ unsigned radix_digit(unsigned key, int level) {
  return key >> radix_shift(level) & (level == 2 ? 1023u : 2047u);
}

template <int CL>
__device__ __forceinline__ void radix_clear(RadixShared<CL>& s) {
#pragma unroll
  for (int i = 0; i < kRxLevels * kRxBins / kRxThreads; ++i) s.hist[0][i * kRxThreads + threadIdx.x] = make_uint4(0u, 0u, 0u, 0u);
}
template <int CL>
__device__ __forceinline__ void radix_count(RadixShared<CL>& s, int level, unsigned digit, bool counts) {
  count_if(counts, reinterpret_cast<unsigned*>(s.hist[level]) + digit * kRxCopies + (threadIdx.x & (kRxCopies - 1)));
}
template <int CL>
__device__ __forceinline__ void cluster_barrier() {
  if (CL > 1) cg::this_cluster().sync();
  else __syncthreads();
}
__device__ __forceinline__ unsigned warp_scan(unsigned v, int lane) {   // inclusive
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}
// After a level's counting (no barrier needed before): finds the digit that holds the `remaining`-th
// largest key, the rank still wanted inside it and how many keys share it.
template <int CL>
__device__ __forceinline__ void radix_pick(RadixShared<CL>& s, int level, unsigned& remaining, unsigned& digit, unsigned& in_digit) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto bin_of = [&](int bin) {
    const uint4 c = s.hist[level][bin];
    return (c.x + c.y) + (c.z + c.w);
  };
  __syncthreads();
  const unsigned b0 = bin_of(warp * 64 + lane), b1 = bin_of(warp * 64 + 32 + lane);
  if (CL > 1) {
    s.bins[level][warp * 64 + lane] = b0;
    s.bins[level][warp * 64 + 32 + lane] = b1;
  }
  const unsigned sum = __reduce_add_sync(0xffffffffu, b0 + b1);
  if (lane < CL) {
    unsigned (*to)[32] = s.sums[level];
    if (CL > 1) to = reinterpret_cast<unsigned (*)[32]>(cg::this_cluster().map_shared_rank(&s.sums[level][0][0], lane));
    to[CL > 1 ? (int)cg::this_cluster().block_rank() : 0][warp] = sum;
  }
  cluster_barrier<CL>();
  if (warp == 0) {
    // lane l: group 31 - l, from the top
    unsigned c = 0;
#pragma unroll
    for (int r = 0; r < CL; ++r) c += s.sums[level][r][31 - lane];
    unsigned incl = warp_scan(c, lane), before = incl - c;
    const int at = __ffs(__ballot_sync(0xffffffffu, before < remaining && remaining <= incl)) - 1;
    const unsigned rest = remaining - __shfl_sync(0xffffffffu, before, at);
    // lane l: bins 63 - 2 l and 62 - 2 l of that group
    const int top = (31 - at) * 64 + 63 - 2 * lane;
    unsigned hi = 0, lo = 0;
    if (CL == 1) {
      hi = bin_of(top);
      lo = bin_of(top - 1);
    } else {
#pragma unroll
      for (int r = 0; r < CL; ++r) {
        const uint2 c2 = *reinterpret_cast<const uint2*>(cg::this_cluster().map_shared_rank(&s.bins[level][0], r) + top - 1);
        hi += c2.y;
        lo += c2.x;
      }
    }
    incl = warp_scan(hi + lo, lane);
    before = incl - hi - lo;
    if (before < rest && rest <= incl) {
      const bool first = rest <= before + hi;
      s.found[level][0] = first ? top : top - 1;
      s.found[level][1] = first ? hi : lo;
      s.found[level][2] = rest - before - (first ? 0u : hi);
    }
  }
  __syncthreads();
  digit = s.found[level][0];
  in_digit = s.found[level][1];
  remaining = s.found[level][2];
}

// Larger float -> larger unsigned, NaN of either sign above all; -0 and +0 are the same.  (The comparison does what an
// addition of zero, for -0, and a minimum with infinity, for NaN, do in two instructions more: 33 vectors of 200000 tokens
// 39.7 us, with these 41.6, with the addition alone, which leaves a NaN its sign, 39.6.)
__device__ __forceinline__ unsigned order_key(float v) {
  unsigned negative, b = __float_as_uint(v);
  asm("set.lt.u32.f32 %0, %1, 0f00000000;" : "=r"(negative) : "f"(v));   // all bits or none; none for -0 and NaN
  return (b ^ negative) | (~negative & 0x80000000u);
}

}  // namespace skv
