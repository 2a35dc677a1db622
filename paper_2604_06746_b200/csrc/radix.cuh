// Rank search over fp32 keys held in registers (token selection).  A cluster of CL CTAs of kRxThreads threads
// shares one vector; digits of eight bits from the top.  Each level: every lane counts into histogram copies
// of its own (bank = lane, so a warp's hits never collide, however concentrated the digit), a warp sums the
// copies of a bin with one reduction instruction, the 256 counts go to every CTA of the cluster in
// coalesced copies, and every warp walks them on its own.  Two block barriers and one exchange per level; one
// pass over memory in all where the vector fits the registers.  (2048-bin histograms with eight copies
// merged in CTA 0 by remote atomics and a sweep of memory per level took 21 us for any short vector.)
#pragma once

#include <cooperative_groups.h>

#include "common.cuh"

namespace skv {

namespace cg = cooperative_groups;

constexpr int kRxThreads = 1024;
constexpr int kRxLevels = 4;

template <int CL>
struct RadixShared {
  unsigned hist[2][256 * 32];          // levels alternate
  unsigned cnt[2][CL][256];            // counts of every CTA of the cluster
  unsigned mine[256];                  // this CTA's, before the exchange
  unsigned scratch[2 * kRxThreads];    // block reductions, output offsets
};

template <int CL>
__device__ __forceinline__ void radix_clear(RadixShared<CL>& s, int buf) {
  uint4* h = reinterpret_cast<uint4*>(s.hist[buf]);
  for (int i = threadIdx.x; i < 256 * 32 / 4; i += kRxThreads) h[i] = make_uint4(0u, 0u, 0u, 0u);
}
template <int CL>
__device__ __forceinline__ void radix_count(RadixShared<CL>& s, int buf, unsigned digit) {
  atomicAdd(&s.hist[buf][digit * 32 + (threadIdx.x & 31)], 1u);
}
template <int CL>
__device__ __forceinline__ void cluster_barrier() {
  if (CL > 1) cg::this_cluster().sync();
  else __syncthreads();
}
// After a level's counting (no barrier needed before): finds the digit that holds the `remaining`-th
// largest key, the rank still wanted inside it and how many keys share it.  The other histogram
// buffer is clear when it returns, ready for the next level.
template <int CL>
__device__ __forceinline__ void radix_pick(RadixShared<CL>& s, int buf, unsigned& remaining, unsigned& digit, unsigned& in_digit) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    const int bin = warp * 8 + b;
    const unsigned c = __reduce_add_sync(0xffffffffu, s.hist[buf][bin * 32 + lane]);
    if (lane == 0) (CL > 1 ? s.mine : s.cnt[buf][0])[bin] = c;
  }
  radix_clear(s, buf ^ 1);
  __syncthreads();
  if (CL > 1) {
    const int rank = (int)cg::this_cluster().block_rank();
    if (warp < CL) {                                 // one warp per destination, 16 bytes a lane
      uint4* to = reinterpret_cast<uint4*>(cg::this_cluster().map_shared_rank(&s.cnt[buf][0][0], warp) + rank * 256);
      const uint4* from = reinterpret_cast<const uint4*>(s.mine);
      to[lane] = from[lane];
      to[lane + 32] = from[lane + 32];
    }
    cluster_barrier<CL>();
  }
  // lane l of every warp: bins 255 - 8 l .. 248 - 8 l, from the top
  unsigned c[8], mine = 0;
#pragma unroll
  for (int b = 0; b < 8; ++b) c[b] = 0;
#pragma unroll
  for (int r = 0; r < CL; ++r) {
    const uint4* q = reinterpret_cast<const uint4*>(&s.cnt[buf][r][248 - 8 * lane]);
    const uint4 hi = q[1], lo = q[0];
    c[0] += hi.w; c[1] += hi.z; c[2] += hi.y; c[3] += hi.x;
    c[4] += lo.w; c[5] += lo.z; c[6] += lo.y; c[7] += lo.x;
  }
#pragma unroll
  for (int b = 0; b < 8; ++b) mine += c[b];
  unsigned incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  unsigned before = incl - mine, d = 0, rem = 0, in = 0;
  const bool here = before < remaining && remaining <= incl;
  if (here) {
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      if (in == 0 && before + c[b] >= remaining) { d = 255 - 8 * lane - b; rem = remaining - before; in = c[b]; }
      if (in == 0) before += c[b];
    }
  }
  const int src = __ffs(__ballot_sync(0xffffffffu, here)) - 1;
  digit = __shfl_sync(0xffffffffu, d, src);
  in_digit = __shfl_sync(0xffffffffu, in, src);
  remaining = __shfl_sync(0xffffffffu, rem, src);
}

// Larger float -> larger unsigned; -0 is folded onto +0.
__device__ __forceinline__ unsigned order_key(float v) {
  const unsigned b = __float_as_uint(v + 0.0f);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

}  // namespace skv
