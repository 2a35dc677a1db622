// Rank search over fp32 keys held in registers, shared by the token selection and the head
// statistics.  A cluster of CL CTAs of kRxThreads threads shares one vector; digits of eight bits from
// the top.  Each level: every lane counts into histogram copies of its own (bank = lane, so a warp's
// hits never collide, however concentrated the digit), a warp sums the copies of a bin with one
// reduction instruction, the 256 counts go to every CTA of the cluster in coalesced copies, and every
// warp walks them on its own.  Two block barriers and one exchange per level; one pass over memory in
// all where the vector fits the registers.  (Before: 2048-bin histograms with eight copies merged in
// CTA 0 by remote atomics, a serial walk over warp totals and a sweep of memory per level: 21 us
// for any short vector, 35 us for a layer's head statistics.)
#pragma once

#include <cooperative_groups.h>

#include "common.cuh"

namespace skv {

namespace cg = cooperative_groups;

constexpr int kRxThreads = 1024;
constexpr int kRxLevels = 4;

// COPIES of a bin; BUFFERS: two alternate from level to level, one costs a barrier more; THREADS of a CTA.
template <int CL_, int COPIES_ = 32, int BUFFERS_ = 2, int THREADS_ = kRxThreads>
struct RadixShared {
  static constexpr int CL = CL_, COPIES = COPIES_, BUFFERS = BUFFERS_, THREADS = THREADS_;
  unsigned hist[BUFFERS][256 * COPIES];
  unsigned cnt[2][CL][256];            // counts of every CTA of the cluster
  unsigned mine[256];                  // this CTA's, before the exchange
  unsigned scratch[THREADS + 64];      // block reductions, output offsets
  float red[4][33];
};
using RadixResident = RadixShared<1, 16, 1>;      // leaves shared memory for the vector itself
using RadixSmall = RadixShared<1, 16, 1, 256>;    // short vectors, many of them: several CTAs on an SM

template <typename S>
__device__ __forceinline__ void radix_clear(S& s, int buf) {
  uint4* h = reinterpret_cast<uint4*>(s.hist[buf % S::BUFFERS]);
  for (int i = threadIdx.x; i < 256 * S::COPIES / 4; i += S::THREADS) h[i] = make_uint4(0u, 0u, 0u, 0u);
}
template <typename S>
__device__ __forceinline__ void radix_count(S& s, int buf, unsigned digit) {
  atomicAdd(&s.hist[buf % S::BUFFERS][digit * S::COPIES + (threadIdx.x & (S::COPIES - 1))], 1u);
}
template <int CL>
__device__ __forceinline__ void cluster_barrier() {
  if (CL > 1) cg::this_cluster().sync();
  else __syncthreads();
}
// After a level's counting (no barrier needed before): finds the digit that holds the `remaining`-th
// largest key, the rank still wanted inside it and how many keys share it.  The histogram of the next
// level is clear when it returns.
template <typename S>
__device__ __forceinline__ void radix_pick(S& s, int buf, unsigned& remaining, unsigned& digit, unsigned& in_digit) {
  constexpr int CL = S::CL, COPIES = S::COPIES;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned* const h = s.hist[buf % S::BUFFERS];
  unsigned* const to_cnt = CL > 1 ? s.mine : s.cnt[buf][0];
  __syncthreads();
  constexpr int kAt = 32 / COPIES;                   // bins a warp sums side by side
  constexpr int kBins = 256 / (S::THREADS / 32);     // bins of a warp
#pragma unroll 8
  for (int b = 0; b < kBins; b += kAt) {
    unsigned c = h[(warp * kBins + b) * COPIES + lane];
    if (COPIES == 32) {
      c = __reduce_add_sync(0xffffffffu, c);
    } else {
#pragma unroll
      for (int o = COPIES / 2; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    if (lane % COPIES == 0) to_cnt[warp * kBins + b + lane / COPIES] = c;
  }
  if (S::BUFFERS == 1) __syncthreads();
  radix_clear(s, buf + 1);
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

// Copies x[0 .. n) to shared memory (dst 16-byte aligned), 16 bytes at a time.
__device__ __forceinline__ void stage_vector(float* dst, const float* __restrict__ x, int n) {
  const int head = min(n, (int)((4 - ((uintptr_t)x >> 2 & 3)) & 3)), n4 = (n - head) / 4;
  if ((int)threadIdx.x < head) dst[threadIdx.x] = x[threadIdx.x];
  const float4* x4 = reinterpret_cast<const float4*>(x + head);
#pragma unroll 4
  for (int i = threadIdx.x; i < n4; i += kRxThreads) {
    const float4 v = x4[i];
    if (head == 0) {
      reinterpret_cast<float4*>(dst)[i] = v;
    } else {
      float* d = dst + head + 4 * i;
      d[0] = v.x; d[1] = v.y; d[2] = v.z; d[3] = v.w;
    }
  }
  for (int i = head + 4 * n4 + threadIdx.x; i < n; i += kRxThreads) dst[i] = x[i];
}
// The longest vector one CTA holds in shared memory beside a RadixResident.
constexpr int kResidentMax = 50 * 1024;
constexpr int kResidentBytes = (int)(sizeof(RadixResident) + 15) / 16 * 16 + kResidentMax * 4;
static_assert(kResidentBytes + 1024 <= 227 * 1024, "shared memory of one CTA");

// Larger float -> larger unsigned; -0 is folded onto +0.
__device__ __forceinline__ unsigned order_key(float v) {
  const unsigned b = __float_as_uint(v + 0.0f);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// Kernel launch with a cluster of CL CTAs and early start.
template <int CL, int THREADS = kRxThreads, typename... KArgs, typename... Args>
inline cudaError_t launch_cluster(void (*kernel)(KArgs...), int grid, size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = CL;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = CL > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

}  // namespace skv
