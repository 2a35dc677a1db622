// Rank search over fp32 keys held in registers (token selection).  A cluster of CL CTAs of kRxThreads threads
// shares one vector; digits of 11, 11 and 10 bits from the top.  Each level: keys are counted into a histogram of
// 2048 bins (four copies of a bin, one for every fourth lane); 32 warps add up 64 bins each, the 32 sums go to every CTA
// of the cluster, and every warp walks them and then the 64 bins that hold the wanted rank on its own; in a cluster,
// where these come through distributed shared memory, one warp does it for its CTA (all 32 of them: 131072 keys 103 us).
// Two or three block barriers a level; one pass over memory in all where the vector fits the registers.
// Bound by the chain of barriers and shared-memory round trips.  Four levels of eight bits with a copy of every bin
// per lane took 7.5 us for 1000 keys (now 5.1), 9.7 for 5003 (6.7), 16.8 for 32768 (9.3), 22.3 for 131072 (18.6).
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
  unsigned sums[kRxLevels][CL][32];    // of 64 bins each, of every CTA of the cluster
  unsigned found[kRxLevels][3];        // clusters: digit, keys in it, rank in it
  unsigned scratch[2 * kRxThreads];    // block reductions, output offsets
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
__device__ __forceinline__ void radix_count(RadixShared<CL>& s, int level, unsigned digit) {
  atomicAdd(reinterpret_cast<unsigned*>(s.hist[level]) + digit * kRxCopies + (threadIdx.x & (kRxCopies - 1)), 1u);
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
  auto bin_of = [&](const uint4* hist, int bin) {
    const uint4 c = hist[bin];
    return (c.x + c.y) + (c.z + c.w);
  };
  __syncthreads();
  const unsigned sum = __reduce_add_sync(0xffffffffu, bin_of(s.hist[level], warp * 64 + lane) + bin_of(s.hist[level], warp * 64 + 32 + lane));
  if (lane < CL) {
    unsigned (*to)[32] = s.sums[level];
    if (CL > 1) to = reinterpret_cast<unsigned (*)[32]>(cg::this_cluster().map_shared_rank(&s.sums[level][0][0], lane));
    to[CL > 1 ? (int)cg::this_cluster().block_rank() : 0][warp] = sum;
  }
  cluster_barrier<CL>();
  if (CL == 1 || warp == 0) {
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
#pragma unroll
    for (int r = 0; r < CL; ++r) {
      const uint4* h = s.hist[level];
      if (CL > 1) h = cg::this_cluster().map_shared_rank(s.hist[level], r);
      hi += bin_of(h, top);
      lo += bin_of(h, top - 1);
    }
    incl = warp_scan(hi + lo, lane);
    before = incl - hi - lo;
    const bool first = rest <= before + hi;
    const int src = __ffs(__ballot_sync(0xffffffffu, before < rest && rest <= incl)) - 1;
    digit = __shfl_sync(0xffffffffu, (unsigned)(first ? top : top - 1), src);
    in_digit = __shfl_sync(0xffffffffu, first ? hi : lo, src);
    remaining = __shfl_sync(0xffffffffu, rest - before - (first ? 0u : hi), src);
  }
  if (CL > 1) {
    if (threadIdx.x == 0) { s.found[level][0] = digit; s.found[level][1] = in_digit; s.found[level][2] = remaining; }
    __syncthreads();
    digit = s.found[level][0];
    in_digit = s.found[level][1];
    remaining = s.found[level][2];
  }
}

// Larger float -> larger unsigned; -0 is folded onto +0.
__device__ __forceinline__ unsigned order_key(float v) {
  const unsigned b = __float_as_uint(v + 0.0f);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

}  // namespace skv
