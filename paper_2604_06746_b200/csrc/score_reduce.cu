// Small deterministic reductions after the scorers: the sum
// over heads with the centrality update, per-head sparsity / variance with the layer's metrics, and
// the closed-form centrality re-accumulation.
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "radix.cuh"

namespace skv {
namespace {

// ---- what follows the scorer passes of a layer, of several layers or of a packed batch ----------
// One launch: CTAs of clusters first (one cluster per (problem, head) vector, Eq. 5-6), then blocks
// that sum 128 x VEC keys over the heads (Eq. 2) and carry the centrality (Eq. 3).  Every sum has a
// fixed order.
struct FinishArgs {
  const float* cols;                   // problem p, head h, key j at cols + p * layer_stride + h * col_stride + j
  long long layer_stride, col_stride;
  int H, n, n_prob;
  float lambda;
  float* s_out;                        // problem p at s_out + p * s_stride
  long long s_stride;
  float* c_inout;                      // layers: one vector carried through them; packed: at s_out's offsets
  int c_from_zero;                     // its old contents count as 0
  const float* row_ent;                // [n_prob][rows_pad], or NULL: no entropy, no sums
  int rows_pad, n_valid;
  float* metrics;                      // [n_prob][3]
  float* head_part;                    // [n_prob][H][4]
  int with_stats, n_stat_ctas, chunks; // chunks: key ranges a problem's sum is cut into
  int* stat_ctr;                       // [n_prob] heads done; zero between launches
  int* chunk_ctr;                      // [chunks] layers done; zero between launches
  int packed;                          // sequences of one layer: problem p owns columns [cu[p], cu[p + 1])
  int cu[kMaxBatch + 1];
};
constexpr int kSumLanes = 128, kSumGroups = 8;

struct Problem { const float* cols; float* s; int n; };
__device__ __forceinline__ Problem problem_of(const FinishArgs& a, int p) {
  if (a.packed) return {a.cols + a.cu[p], a.s_out + a.cu[p], a.cu[p + 1] - a.cu[p]};
  return {a.cols + (size_t)p * a.layer_stride, a.s_out + (size_t)p * a.s_stride, a.n};
}

// Sum of v over the block, in every thread of warp 0 (fixed order).
__device__ __forceinline__ float block_total(float v, float* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) red[warp] = v;
  __syncthreads();
  if (warp == 0) {
    v = lane < (int)(blockDim.x >> 5) ? red[lane] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  }
  return v;
}

template <int VEC> struct Keys;
template <> struct Keys<4> { using T = float4; };
template <> struct Keys<1> { using T = float; };
__device__ __forceinline__ float4 decay(float l, const float4& c, const float4& s) {
  return make_float4(fmaf(l, c.x, s.x), fmaf(l, c.y, s.y), fmaf(l, c.z, s.z), fmaf(l, c.w, s.w));
}
__device__ __forceinline__ float decay(float l, float c, float s) { return fmaf(l, c, s); }

template <int VEC>
struct SumShared {
  typename Keys<VEC>::T part[kSumGroups - 1][kSumLanes];
  float red[32];
  int last;
};
// Keys [chunk * 128 * VEC, ...) of problem p: eight groups of heads side by side (one chain of H loads
// took 9 us), their sums added in group order.  The centrality of several layers is a recursion over
// them: the block that completes a key range takes all of its layers.
// THREADS: each row of 128 threads takes kSumGroups * 128 / THREADS of the groups.
template <int VEC, int THREADS>
__device__ __forceinline__ void sum_block(const FinishArgs& a, SumShared<VEC>& sh, int p, int chunk) {
  using T = typename Keys<VEC>::T;
  auto& part = sh.part;
  float* const red = sh.red;
  int& last = sh.last;
  const Problem pb = problem_of(a, p);
  constexpr int kRows = THREADS / kSumLanes, kMine = kSumGroups / kRows;
  const int lane_j = threadIdx.x & (kSumLanes - 1), grp = threadIdx.x / kSumLanes;
  const int j = (chunk * kSumLanes + lane_j) * VEC;    // VEC 4: every problem's n is a multiple of 4
  const int h_per = (a.H + kSumGroups - 1) / kSumGroups;
  T s{};
#pragma unroll
  for (int m = 0; m < kMine; ++m) {
    const int gr = grp + m * kRows, h_lo = min(a.H, gr * h_per), h_hi = min(a.H, h_lo + h_per);
    T t{};
    if (j < pb.n) {
#pragma unroll 4
      for (int h = h_lo; h < h_hi; ++h) add_to(t, *reinterpret_cast<const T*>(pb.cols + (size_t)h * a.col_stride + j));
    }
    if (gr == 0) s = t;
    else part[gr - 1][lane_j] = t;
  }
  __syncthreads();
  if (grp == 0 && j < pb.n) {
#pragma unroll
    for (int k = 0; k < kSumGroups - 1; ++k) add_to(s, part[k][lane_j]);
    *reinterpret_cast<T*>(pb.s + j) = s;
  }
  if (a.c_inout) {
    const bool chained = !a.packed && a.n_prob > 1;
    T* c = reinterpret_cast<T*>(a.c_inout + (a.packed ? a.cu[p] : 0) + j);
    if (!chained) {
      if (grp == 0 && j < pb.n) *c = a.c_from_zero ? s : decay(a.lambda, *c, s);
    } else {
      __threadfence();
      __syncthreads();
      if (threadIdx.x == 0) last = atomicAdd(&a.chunk_ctr[chunk], 1) == a.n_prob - 1;
      __syncthreads();
      if (last) {
        __threadfence();
        if (grp == 0 && j < pb.n) {
          T acc{};
          if (!a.c_from_zero) acc = *c;
#pragma unroll 8
          for (int l = 0; l < a.n_prob; ++l)
            acc = decay(a.lambda, acc, __ldcg(reinterpret_cast<const T*>(a.s_out + (size_t)l * a.s_stride + j)));
          *c = acc;
        }
        if (threadIdx.x == 0) a.chunk_ctr[chunk] = 0;
      }
    }
  }
  if (chunk != 0) return;
  // the problem's entropy (Eq. 4); rows that do not exist hold 0
  float ent = 0.f;
  // (the same partial sums whatever the block size: thread t of 1024 takes rows t, t + 1024, ...)
  for (int t = threadIdx.x; t < kRxThreads; t += THREADS) {
    float e = 0.f;
    for (int r = t; r < a.rows_pad; r += kRxThreads) e += a.row_ent[(size_t)p * a.rows_pad + r];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if ((t & 31) == 0) red[t >> 5] = e;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    ent = red[threadIdx.x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ent += __shfl_xor_sync(0xffffffffu, ent, o);
  }
  if (threadIdx.x == 0) {
    a.metrics[p * 3] = ent / (float)a.n_valid;
    if (!a.with_stats) a.metrics[p * 3 + 1] = a.metrics[p * 3 + 2] = __int_as_float(0x7fc00000);
  }
}

// Eq. 5 and 6 of one (problem, head) vector, by a cluster or by one CTA: the sum of squared deviations
// from 1/n (the pooled vector sums to 1, so 1/n is its mean; summing deviations instead of squares
// keeps near-uniform attention from cancelling) and the mass of the floor(n / 10) largest entries.
// Three radix levels give the threshold to 24 bits; of the entries that share them, the ones still
// wanted count with their average; a level that settles it is the last.  All entries are >= 0: the
// order of the bit patterns is theirs.
template <int ITEMS, typename S>
__device__ __forceinline__ void stats_cta(const FinishArgs& a, S& s, float* vec_s, int vec) {
  constexpr int CL = S::CL;
  constexpr bool RESIDENT = std::is_same_v<S, RadixResident>;
  const int tid = threadIdx.x;
  const int rank = CL > 1 ? (int)cg::this_cluster().block_rank() : 0;
  const int p = vec / a.H;
  const Problem pb = problem_of(a, p);
  const float* x = pb.cols + (size_t)(vec - p * a.H) * a.col_stride;
  const int n = pb.n, per = (n + CL - 1) / CL, lo = min(n, rank * per), hi = min(n, lo + per);
  constexpr int kChunk = S::THREADS * ITEMS;
  const int chunks = (per + kChunk - 1) / kChunk;
  unsigned key[ITEMS];
  auto load = [&](int c) {
#pragma unroll
    for (int e = 0; e < ITEMS; ++e) {
      const int j = lo + c * kChunk + e * S::THREADS + tid;
      key[e] = j < hi ? __float_as_uint((RESIDENT ? vec_s[j] : x[j]) + 0.f) : 0x80000000u;   // sign bit: no entry (-0 becomes +0)
    }
  };
  if (RESIDENT) {
    stage_vector(vec_s, x, n);
    __syncthreads();
  }
  const float mean = 1.f / (float)n;
  float sq = 0.f;
  unsigned remaining = (unsigned)max(1, n / 10), thr = 0, in = 0, known = 0;   // known: mask of the bits found so far
#pragma unroll 1
  for (int level = 0; level < 3; ++level) {
    const int shift = 24 - 8 * level;
    const unsigned mask = level == 0 ? 0x80000000u : 0xffffffffu << (shift + 8);
    for (int c = 0; c < chunks; ++c) {
      if (chunks > 1 || level == 0) load(c);
#pragma unroll
      for (int e = 0; e < ITEMS; ++e) {
        if (level == 0 && !(key[e] >> 31)) {
          const float dv = __uint_as_float(key[e]) - mean;
          sq = fmaf(dv, dv, sq);
        }
        if ((key[e] & mask) == thr) radix_count(s, level & 1, (key[e] >> shift) & 255u);
      }
    }
    unsigned digit;
    radix_pick(s, level & 1, remaining, digit, in);
    thr |= digit << shift;
    known = 0xffffffffu << shift;
    if (in == remaining) break;                      // all entries that share these bits count
  }
  float above = 0.f, inside = 0.f;
  for (int c = 0; c < chunks; ++c) {
    if (chunks > 1) load(c);
#pragma unroll
    for (int e = 0; e < ITEMS; ++e) {
      const unsigned top = key[e] & known;
      if (!(key[e] >> 31)) {
        if (top > thr) above += __uint_as_float(key[e]);
        else if (top == thr) inside += __uint_as_float(key[e]);
      }
    }
  }
  sq = block_total(sq, s.red[0]);
  above = block_total(above, s.red[1]);
  inside = block_total(inside, s.red[2]);
  __shared__ float slots[3 * CL];
  if (CL > 1) {
    if (tid == 0) {
      float* to = cg::this_cluster().map_shared_rank(slots, 0);
      to[3 * rank] = sq; to[3 * rank + 1] = above; to[3 * rank + 2] = inside;
    }
    cluster_barrier<CL>();
    if (rank != 0) return;
  }
  if (tid >= 32) return;
  int last = 0;
  if (tid == 0) {
    if (CL > 1) {
      sq = above = inside = 0.f;
      for (int r = 0; r < CL; ++r) { sq += slots[3 * r]; above += slots[3 * r + 1]; inside += slots[3 * r + 2]; }
    }
    float* hp = a.head_part + (size_t)vec * 4;
    __stcg(hp, sq);
    __stcg(hp + 1, above + (float)remaining * (inside / (float)in));
    __threadfence();
    last = atomicAdd(&a.stat_ctr[p], 1) == a.H - 1;
  }
  if (!__shfl_sync(0xffffffffu, last, 0)) return;
  // the last head of the problem averages all of them (fixed order)
  __threadfence();
  float rho = 0.f, var = 0.f;
  for (int h = tid; h < a.H; h += 32) {
    const float* hp = a.head_part + ((size_t)p * a.H + h) * 4;
    var += __ldcg(hp) * mean;
    rho += __ldcg(hp + 1);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    rho += __shfl_xor_sync(0xffffffffu, rho, o);
    var += __shfl_xor_sync(0xffffffffu, var, o);
  }
  if (tid == 0) {
    a.metrics[p * 3 + 1] = rho / (float)a.H;
    a.metrics[p * 3 + 2] = var / (float)a.H;
    a.stat_ctr[p] = 0;
  }
}

template <int ITEMS, int VEC, typename S>
__global__ void
__launch_bounds__(S::THREADS, S::THREADS < kRxThreads ? 4 : ITEMS <= 8 && !std::is_same_v<S, RadixResident> ? 2 : 1)
finish(const __grid_constant__ FinishArgs a) {
  extern __shared__ __align__(16) unsigned char fin_smem[];
  S& s = *reinterpret_cast<S*>(fin_smem);
  const bool stats = (int)blockIdx.x < a.n_stat_ctas;
  pdl_trigger();
  if (stats) {
    radix_clear(s, 0);
    cluster_barrier<S::CL>();                        // all CTAs of the cluster run before any remote access
  }
  pdl_wait();
  if (stats) {
    stats_cta<ITEMS>(a, s, reinterpret_cast<float*>(fin_smem + (sizeof(S) + 15) / 16 * 16), blockIdx.x / S::CL);
  } else {
    const int b = blockIdx.x - a.n_stat_ctas, p = b / a.chunks;
    if (p < a.n_prob) sum_block<VEC, S::THREADS>(a, *reinterpret_cast<SumShared<VEC>*>(fin_smem), p, b - p * a.chunks);
  }
}
constexpr int kSumThreads = 256;     // many short blocks: 16 loads in flight per thread
template <int VEC>
__global__ void __launch_bounds__(kSumThreads) sum_layers(const __grid_constant__ FinishArgs a) {
  __shared__ SumShared<VEC> sh;
  pdl_trigger();
  pdl_wait();
  sum_block<VEC, kSumThreads>(a, sh, blockIdx.x / a.chunks, blockIdx.x % a.chunks);
}

// ---- Eq. 5-6 of many long vectors: one CTA per vector, two sweeps over memory --------------------
// With more vectors than the clusters above could run side by side (32 layers of 131072 keys: 1024
// vectors, 231 us in two sweeps of 537 MB; clusters of eight 1630 us).  Counting sweeps locate the
// k-th largest value to 22 bits:
//   sweep 1: histogram of bits 30..20 (exponent + 3 mantissa bits); sum of squared deviations
//   sweep 2: exact sum of the entries above the threshold bin and a histogram of bits 19..9 inside it
// The entries inside the threshold bin are then summed as count x bin midpoint: bins of the second
// level are 2^-14 wide relative to their value, far inside the metric's tolerance.
constexpr int kHsThreads = 1024, kHsBins = 2048;
constexpr int kHsCopies = 16;      // copies of a bin, so that a warp's hits on one bin spread

// Applies f to a[lo .. hi) once each, kHsThreads threads together: 16-byte loads, four of them in
// flight per thread, scalar accesses only for the unaligned ends.  The order in which a thread
// meets its entries is fixed.
template <class F>
__device__ __forceinline__ void sweep_from_memory(const float* __restrict__ a, int lo, int hi, int tid, F f) {
  const int mis = (int)((reinterpret_cast<uintptr_t>(a + lo) >> 2) & 3u);
  const int n_head = min(hi - lo, (4 - mis) & 3);
  if (tid < n_head) f(a[lo + tid]);
  const int b0 = lo + n_head;
  const int n4 = (hi - b0) >> 2;
  const float4* a4 = reinterpret_cast<const float4*>(a + b0);
  int i = tid;
  for (; i + 3 * kHsThreads < n4; i += 4 * kHsThreads) {
    const float4 v0 = a4[i], v1 = a4[i + kHsThreads], v2 = a4[i + 2 * kHsThreads], v3 = a4[i + 3 * kHsThreads];
    f(v0.x); f(v0.y); f(v0.z); f(v0.w);
    f(v1.x); f(v1.y); f(v1.z); f(v1.w);
    f(v2.x); f(v2.y); f(v2.z); f(v2.w);
    f(v3.x); f(v3.y); f(v3.z); f(v3.w);
  }
  for (; i < n4; i += kHsThreads) {
    const float4 v = a4[i];
    f(v.x); f(v.y); f(v.z); f(v.w);
  }
  const int t0 = b0 + 4 * n4;
  if (t0 + tid < hi) f(a[t0 + tid]);
}

// Called by all threads of a 1024-thread block after a histogram pass over `nb` = 2048 bins.
// Walks the bins from the top and finds the bin holding the `remaining`-th largest candidate;
// writes that bin and the rank still wanted inside it.  `scratch` holds 33 words.
__device__ __forceinline__ void block_pick_from_top(const unsigned* hist, unsigned remaining,
                                                    unsigned* scratch, unsigned* sel_bin, unsigned* sel_rem) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b_hi = 2047 - 2 * tid, b_lo = b_hi - 1;        // this thread's two bins, higher first
  const unsigned c_hi = hist[b_hi], c_lo = hist[b_lo];
  const unsigned mine = c_hi + c_lo;
  unsigned incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  __syncthreads();
  if (lane == 31) scratch[warp] = incl;
  __syncthreads();
  unsigned before = incl - mine;
  for (int w = 0; w < warp; ++w) before += scratch[w];
  if (before < remaining && remaining <= before + mine) {
    if (before + c_hi >= remaining) { *sel_bin = (unsigned)b_hi; *sel_rem = remaining - before; }
    else { *sel_bin = (unsigned)b_lo; *sel_rem = remaining - before - c_hi; }
  }
  __syncthreads();
}

// Shared memory: hist[kHsBins][kHsCopies] | merged[2][kHsBins] (dynamic, 144 KB).
__global__ void __launch_bounds__(kHsThreads)
head_stats(const float* __restrict__ cols, long long layer_stride, long long col_stride, int H, int n, int k_rho,
           float* __restrict__ head_part) {
  extern __shared__ unsigned hs_smem[];
  unsigned* hist = hs_smem;
  unsigned* merged = hs_smem + kHsBins * kHsCopies;
  __shared__ float red[3][33];
  __shared__ unsigned scan_tmp[33];
  __shared__ unsigned sel_bin, sel_rem;
  const int head = blockIdx.x;                       // (layer, head) pair
  const float* a = cols + (size_t)(head / H) * layer_stride + (size_t)(head % H) * col_stride;
  const int tid = threadIdx.x, copy = tid & (kHsCopies - 1);
  auto clear_local = [&]() {
    for (int b = tid; b < kHsBins * kHsCopies; b += kHsThreads) hist[b] = 0;
  };
  auto push = [&](int level) {                       // sum of a bin's copies
    for (int b = tid; b < kHsBins; b += kHsThreads) {
      unsigned c = 0;
#pragma unroll
      for (int k = 0; k < kHsCopies; ++k) c += hist[b * kHsCopies + ((k + tid) & (kHsCopies - 1))];   // rotated: no bank conflicts
      merged[level * kHsBins + b] = c;
    }
  };
  pdl_trigger();
  clear_local();
  pdl_wait();                                        // the pooled columns come from the kernels before
  __syncthreads();
  float sq = 0.f;
  const float mean = 1.f / (float)n;
  sweep_from_memory(a, 0, n, tid, [&](float v) {
    const float dv = v - mean;
    sq = fmaf(dv, dv, sq);
    atomicAdd(&hist[((__float_as_uint(v) >> 20) & 0x7ffu) * kHsCopies + copy], 1u);
  });
  __syncthreads();
  push(0);
  __syncthreads();
  clear_local();
  block_pick_from_top(merged, (unsigned)k_rho, scan_tmp, &sel_bin, &sel_rem);
  const unsigned b1 = sel_bin, rem1 = sel_rem;
  float mass = 0.f;
  sweep_from_memory(a, 0, n, tid, [&](float v) {
    const unsigned u = __float_as_uint(v), top = (u >> 20) & 0x7ffu;
    if (top > b1) mass += v;
    else if (top == b1) atomicAdd(&hist[((u >> 9) & 0x7ffu) * kHsCopies + copy], 1u);
  });
  __syncthreads();
  push(1);
  __syncthreads();
  const unsigned* m2 = merged + kHsBins;
  block_pick_from_top(m2, rem1, scan_tmp, &sel_bin, &sel_rem);
  const unsigned b2 = sel_bin, rem2 = sel_rem;
  // entries of the threshold bin above sub-bin b2, and rem2 entries of sub-bin b2 itself
  float in_bin = 0.f;
  for (int b = tid; b < kHsBins; b += kHsThreads) {
    const float mid = __uint_as_float((b1 << 20) | ((unsigned)b << 9) | 0x100u);
    const unsigned cnt = (unsigned)b > b2 ? m2[b] : ((unsigned)b == b2 ? rem2 : 0u);
    in_bin = fmaf((float)cnt, mid, in_bin);
  }
  sq = block_total(sq, red[0]);
  mass = block_total(mass, red[1]);
  in_bin = block_total(in_bin, red[2]);
  if (tid == 0) {
    head_part[head * 4 + 0] = sq;
    head_part[head * 4 + 1] = mass + in_bin;
  }
}

// Eq. 5-6 of a batch of layers from their per-head parts: one thread per layer.
__global__ void head_metrics(const float* __restrict__ head_part, int n_layers, int H, int n,
                             float* __restrict__ metrics) {
  pdl_trigger();
  pdl_wait();
  const int l = blockIdx.x * blockDim.x + threadIdx.x;
  if (l >= n_layers) return;
  float rho = 0.f, var = 0.f;
  const float inv_n = 1.f / (float)n;
  for (int h = 0; h < H; ++h) {
    rho += head_part[((size_t)l * H + h) * 4 + 1];
    var += head_part[((size_t)l * H + h) * 4 + 0] * inv_n;
  }
  metrics[l * 3 + 1] = rho / (float)H;
  metrics[l * 3 + 2] = var / (float)H;
}

// c_out[j] = sum_{l <= pivot} lambda^(pivot - l) s_hist[l][j], as the recursion c = lambda c + s; the loads of
// eight layers are in flight together.
template <int VEC>
__global__ void __launch_bounds__(128) accumulate(const float* __restrict__ s_hist, long long row_stride, int pivot, int n,
                                                  float lambda, float* __restrict__ c_out) {
  using T = typename Keys<VEC>::T;
  pdl_trigger();
  pdl_wait();
  const int j = (blockIdx.x * blockDim.x + threadIdx.x) * VEC;
  if (j >= n) return;
  T c{};
#pragma unroll 8
  for (int l = 0; l <= pivot; ++l) c = decay(lambda, c, *reinterpret_cast<const T*>(s_hist + (size_t)l * row_stride + j));
  *reinterpret_cast<T*>(c_out + j) = c;
}

// Eq. 7-9, then the same recursion.  Every block finds the pivot for itself (one warp, 2 us), so that no
// launch and no host round trip comes between the metrics and the centrality.
template <int VEC>
__global__ void __launch_bounds__(128)
accumulate_at_pivot(const float* __restrict__ s_hist, long long row_stride, int n_layers, int n, float lambda,
                    const float* __restrict__ metrics, float3 weights, int l_limit, float* __restrict__ c_out,
                    volatile int* host, int tag) {
  using T = typename Keys<VEC>::T;
  __shared__ int pivot_s;
  pdl_trigger();
  pdl_wait();
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    constexpr int kPer = kMaxStatLayers / 32;
    double Tl[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) Tl[k] = 0.0;
    for (int col = 0; col < 3; ++col) {
      const double sign = col == 0 ? -1.0 : 1.0, w = col == 0 ? weights.x : col == 1 ? weights.y : weights.z;
      double d[kPer], lo = INFINITY, hi = -INFINITY;
      int nan = 0;
#pragma unroll
      for (int k = 0; k < kPer; ++k) {
        const int l = lane + 32 * k;
        if (l < n_layers) {
          const float m = metrics[l * 3 + col], before = l > 0 ? metrics[(l - 1) * 3 + col] : 0.f;
          nan |= isnan(m);
          d[k] = sign * ((double)m - (double)before);
          if (l > 0) { lo = d[k] < lo ? d[k] : lo; hi = d[k] > hi ? d[k] : hi; }
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const double a = __shfl_xor_sync(0xffffffffu, lo, o), b = __shfl_xor_sync(0xffffffffu, hi, o);
        lo = a < lo ? a : lo;
        hi = b > hi ? b : hi;
      }
      if (__any_sync(0xffffffffu, nan) || !(hi > lo)) continue;
#pragma unroll
      for (int k = 0; k < kPer; ++k) {
        const int l = lane + 32 * k;
        if (l > 0 && l < n_layers)
          Tl[k] = __dadd_rn(Tl[k], __ddiv_rn(__dmul_rn(w, __dsub_rn(d[k], lo)), __dsub_rn(hi, lo)));
      }
    }
    double best = -INFINITY;
    int at = kMaxStatLayers;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int l = lane + 32 * k;
      if (l > 0 && l < n_layers && Tl[k] > best) { best = Tl[k]; at = l; }
      if (blockIdx.x == 0 && l < n_layers) {
        host[1 + l] = __float_as_int((float)Tl[k]);
        __threadfence_system();
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double b = __shfl_xor_sync(0xffffffffu, best, o);
      const int i = __shfl_xor_sync(0xffffffffu, at, o);
      if (b > best || (b == best && i < at)) { best = b; at = i; }
    }
    if (at == kMaxStatLayers) at = n_layers >= 2 ? 1 : 0;   // one layer, or nothing compares
    if (n_layers >= 2 && l_limit >= 0 && at > l_limit) at = l_limit;
    __syncwarp();
    if (lane == 0) {
      pivot_s = at;
      if (blockIdx.x == 0) {                           // last: the host polls this word
        __threadfence_system();
        host[0] = tag | at;
      }
    }
  }
  __syncthreads();
  const int pivot = pivot_s;
  const int j = (blockIdx.x * blockDim.x + threadIdx.x) * VEC;
  if (j >= n) return;
  T c{};
#pragma unroll 8
  for (int l = 0; l <= pivot; ++l) c = decay(lambda, c, *reinterpret_cast<const T*>(s_hist + (size_t)l * row_stride + j));
  *reinterpret_cast<T*>(c_out + j) = c;
}

}  // namespace

// Raises a kernel's shared-memory limit once per device.
template <typename K>
static cudaError_t allow_smem(K* kernel, int bytes, std::atomic<unsigned long long>& ready) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (dev & 63);
  if (ready.load(std::memory_order_acquire) & bit) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) ready.fetch_or(bit, std::memory_order_release);
  return e;
}

template <int CL, int ITEMS, int VEC, typename S = RadixShared<CL>>
static cudaError_t launch_finish_as(FinishArgs& a, int sums, cudaStream_t st) {
  static std::atomic<unsigned long long> ready{0};
  constexpr int smem = std::is_same_v<S, RadixResident> ? kResidentBytes : (int)std::max(sizeof(S), sizeof(SumShared<VEC>));
  const cudaError_t e = allow_smem(finish<ITEMS, VEC, S>, smem, ready);
  if (e != cudaSuccess) return e;
  a.n_stat_ctas = a.n_prob * a.H * CL;
  return launch_cluster<CL, S::THREADS>(finish<ITEMS, VEC, S>, (a.n_stat_ctas + sums + CL - 1) / CL * CL, smem, st, a);
}
template <int VEC>
static cudaError_t launch_finish(FinishArgs& a, int longest, int sms, cudaStream_t st) {
  a.chunks = (longest + kSumLanes * VEC - 1) / (kSumLanes * VEC);
  const int sums = a.row_ent ? a.n_prob * a.chunks : 0;
  if (!a.with_stats) return launch_pdl(sum_layers<VEC>, dim3(sums), dim3(kSumThreads), 0, st, a);
  // More vectors than SMs: four small CTAs share an SM, where those of 1024 threads ran one or two at a time
  // (1024 vectors of 600 / 1777 / 5003 / 8192 keys: 37.6 / 41.3 / 49.0 / 52.6 us before, 21.4 / 23.5 / 33.2 /
  // 36.5 now).  Longer vectors do not fit their registers.
  const int vecs = a.n_prob * a.H;
  if (vecs > sms && longest <= 32 * RadixSmall::THREADS) {
    if (longest <= 8 * RadixSmall::THREADS) return launch_finish_as<1, 8, VEC, RadixSmall>(a, sums, st);
    if (longest <= 16 * RadixSmall::THREADS) return launch_finish_as<1, 16, VEC, RadixSmall>(a, sums, st);
    return launch_finish_as<1, 32, VEC, RadixSmall>(a, sums, st);
  }
  // About one vector per SM: the vector in shared memory.  Clusters would leave some of them for a second
  // wave, and half an SM holds fewer loads in flight (128 vectors of 1777 / 5003 / 20000 / 50000 keys: 13.6 /
  // 15.6 / 30.4 / 67.4 us before, 10.7 / 11.3 / 17.3 / 29.2 now; at 12000 14.2 against the 12.9 of 16 items).
  // With 32 vectors the clusters' extra SMs count for more: 20.7 against 16.5 us at 32768 keys.
  if (2 * vecs > sms && vecs <= sms && longest <= kResidentMax &&
      (longest <= 8 * kRxThreads || longest > 16 * kRxThreads))
    return launch_finish_as<1, 8, VEC, RadixResident>(a, sums, st);
  // one CTA per vector while its registers hold it (no exchange between CTAs), else the smallest
  // cluster that does
  if (longest <= 4 * kRxThreads) return launch_finish_as<1, 4, VEC>(a, sums, st);
  if (longest <= 8 * kRxThreads) return launch_finish_as<1, 8, VEC>(a, sums, st);
  if (longest <= 16 * kRxThreads) return launch_finish_as<1, 16, VEC>(a, sums, st);
  if (longest <= 32 * kRxThreads) return launch_finish_as<2, 16, VEC>(a, sums, st);
  if (longest <= 64 * kRxThreads) return launch_finish_as<4, 16, VEC>(a, sums, st);
  return launch_finish_as<4, 32, VEC>(a, sums, st);
}

static FinishArgs finish_args(const Ctx& ctx, const float* cols, long long col_stride, int n, float* metrics) {
  FinishArgs a = {};
  a.cols = cols; a.col_stride = col_stride;
  a.H = ctx.cfg.n_q_heads; a.n = n; a.n_prob = 1;
  a.rows_pad = ctx.rows_pad; a.n_valid = ctx.rows;
  a.metrics = metrics;
  a.head_part = ctx.ws.head_part; a.stat_ctr = ctx.ws.stat_ctr; a.chunk_ctr = ctx.ws.chunk_ctr;
  return a;
}

cudaError_t launch_finish_layers(const Ctx& ctx, const float* cols, long long layer_stride, long long col_stride, int n,
                                 int n_layers, float lambda, float* s_out, long long s_stride, float* c_inout,
                                 const float* row_ent, bool with_head_stats, float* metrics, cudaStream_t st,
                                 bool c_from_zero) {
  FinishArgs a = finish_args(ctx, cols, col_stride, n, metrics);
  a.layer_stride = layer_stride; a.n_prob = n_layers; a.lambda = lambda; a.c_from_zero = c_from_zero;
  a.s_out = s_out; a.s_stride = s_stride; a.c_inout = c_inout; a.row_ent = row_ent;
  a.with_stats = with_head_stats;
  const bool vec = n % 4 == 0 && col_stride % 4 == 0 && layer_stride % 4 == 0 && s_stride % 4 == 0 &&
                   ((uintptr_t)cols % 16) == 0 && ((uintptr_t)s_out % 16) == 0 && ((uintptr_t)c_inout % 16) == 0;
  return vec ? launch_finish<4>(a, n, ctx.sm_count, st) : launch_finish<1>(a, n, ctx.sm_count, st);
}

cudaError_t launch_finish_packed(const Ctx& ctx, const float* cols, long long col_stride, const int* cu_seqlens, int batch,
                                 float lambda, float* s_out, float* c_inout, const float* row_ent, float* head_part,
                                 bool with_head_stats, float* metrics, cudaStream_t st) {
  FinishArgs a = finish_args(ctx, cols, col_stride, 0, metrics);
  a.n_prob = batch; a.lambda = lambda; a.s_out = s_out; a.c_inout = c_inout; a.row_ent = row_ent;
  a.head_part = head_part; a.with_stats = with_head_stats; a.packed = 1;
  int longest = 0;
  bool vec = col_stride % 4 == 0 && ((uintptr_t)cols % 16) == 0 && ((uintptr_t)s_out % 16) == 0 && ((uintptr_t)c_inout % 16) == 0;
  for (int b = 0; b <= batch; ++b) {
    a.cu[b] = cu_seqlens[b];
    vec = vec && cu_seqlens[b] % 4 == 0;
    if (b > 0) longest = cu_seqlens[b] - cu_seqlens[b - 1] > longest ? cu_seqlens[b] - cu_seqlens[b - 1] : longest;
  }
  return vec ? launch_finish<4>(a, longest, ctx.sm_count, st) : launch_finish<1>(a, longest, ctx.sm_count, st);
}

// Two sweeps per vector where the vectors fill the GPU several times over and are long: with 1024
// vectors 85 / 115 / 231 us at 16000 / 32768 / 131072 keys, the register form 91 / 140 / > 500.
bool head_stats_ride_along(const Ctx& ctx, int n_layers, int n) {
  return (long long)n_layers * ctx.cfg.n_q_heads < 2ll * ctx.sm_count || n <= 8 * kRxThreads;
}

cudaError_t launch_head_stats_batch(const Ctx& ctx, const float* cols, long long layer_stride, long long col_stride,
                                    int n_layers, int n, float* metrics, cudaStream_t st) {
  const int H = ctx.cfg.n_q_heads;
  if (!head_stats_ride_along(ctx, n_layers, n)) {
    static std::atomic<unsigned long long> ready{0};
    const int smem = (kHsBins * kHsCopies + 2 * kHsBins) * (int)sizeof(unsigned);
    cudaError_t e = allow_smem(head_stats, smem, ready);
    if (e != cudaSuccess) return e;
    e = launch_pdl(head_stats, dim3(n_layers * H), dim3(kHsThreads), smem, st, cols, layer_stride, col_stride, H, n,
                   n / 10 < 1 ? 1 : n / 10, ctx.ws.head_part);
    if (e != cudaSuccess) return e;
    return launch_pdl(head_metrics, dim3((n_layers + 63) / 64), dim3(64), 0, st, (const float*)ctx.ws.head_part, n_layers,
                      H, n, metrics);
  }
  FinishArgs a = finish_args(ctx, cols, col_stride, n, metrics);
  a.layer_stride = layer_stride; a.n_prob = n_layers; a.with_stats = 1;
  return launch_finish<1>(a, n, ctx.sm_count, st);
}

cudaError_t launch_accumulate(const float* s_hist, long long row_stride, int pivot, int n,
                              float lambda, float* c_out, cudaStream_t st) {
  if (n % 4 == 0 && row_stride % 4 == 0 && (uintptr_t)s_hist % 16 == 0 && (uintptr_t)c_out % 16 == 0)
    return launch_pdl(accumulate<4>, dim3((n / 4 + 127) / 128), dim3(128), 0, st, s_hist, row_stride, pivot, n, lambda, c_out);
  return launch_pdl(accumulate<1>, dim3((n + 127) / 128), dim3(128), 0, st, s_hist, row_stride, pivot, n, lambda, c_out);
}

cudaError_t launch_accumulate_at_pivot(const float* s_hist, long long row_stride, int n_layers, int n, float lambda,
                                       const float* metrics, const float* weights, int l_limit, float* c_out, int* host,
                                       int tag, cudaStream_t st) {
  const float3 w = make_float3(weights[0], weights[1], weights[2]);
  if (n % 4 == 0 && row_stride % 4 == 0 && (uintptr_t)s_hist % 16 == 0 && (uintptr_t)c_out % 16 == 0)
    return launch_pdl(accumulate_at_pivot<4>, dim3((n / 4 + 127) / 128), dim3(128), 0, st, s_hist, row_stride, n_layers, n,
                      lambda, metrics, w, l_limit, c_out, (volatile int*)host, tag);
  return launch_pdl(accumulate_at_pivot<1>, dim3((n + 127) / 128), dim3(128), 0, st, s_hist, row_stride, n_layers, n, lambda,
                    metrics, w, l_limit, c_out, (volatile int*)host, tag);
}

}  // namespace skv
