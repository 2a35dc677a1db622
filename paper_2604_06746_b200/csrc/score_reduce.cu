// Small deterministic reductions after the scorers: the sum
// over heads with the centrality update, per-head sparsity / variance with the layer's metrics, and
// the closed-form centrality re-accumulation.
#include <cooperative_groups.h>

#include "common.cuh"

namespace skv {
namespace cg = cooperative_groups;
namespace {

// ---- what follows the scorer passes of a layer, of several layers or of a packed batch ----------
// One launch: a CTA or a cluster per (problem, head) vector (Eq. 5-6), and blocks that sum 128 x VEC keys over the
// heads (Eq. 2) and carry the centrality (Eq. 3); which come first is the launch's choice.  Every sum has a fixed order.
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
  int with_stats, chunks;              // chunks: key ranges a problem's sum is cut into
  int stat_ctas;                       // CTAs of a problem's statistics
  int* stat_ctr;                       // [n_prob] heads done; zero between launches
  int* chunk_ctr;                      // [chunks] layers done; zero between launches
  int packed;                          // sequences of one layer: problem p owns columns [cu[p], cu[p + 1])
  int cu[kMaxBatch + 1];
};
constexpr int kSumLanes = 128, kSumGroups = 8;
constexpr int kEntThreads = 1024;      // partial sums of a problem's entropy

struct Problem { const float* cols; float* s; int n; };
__device__ __forceinline__ Problem problem_of(const FinishArgs& a, int p) {
  if (a.packed) return {a.cols + a.cu[p], a.s_out + a.cu[p], a.cu[p + 1] - a.cu[p]};
  return {a.cols + (size_t)p * a.layer_stride, a.s_out + (size_t)p * a.s_stride, a.n};
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
  for (int t = threadIdx.x; t < kEntThreads; t += THREADS) {
    float e = 0.f;
    for (int r = t; r < a.rows_pad; r += kEntThreads) e += a.row_ent[(size_t)p * a.rows_pad + r];
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

// A vector's sums are known (to thread 0; one warp calls): the last head of a problem averages all of them,
// in a fixed order.
__device__ __forceinline__ void head_done(const FinishArgs& a, int vec, float mean, float sq, float mass) {
  const int tid = threadIdx.x, p = vec / a.H;
  int last = 0;
  if (tid == 0) {
    float* hp = a.head_part + (size_t)vec * 4;
    __stcg(hp, sq);
    __stcg(hp + 1, mass);
    __threadfence();
    last = atomicAdd(&a.stat_ctr[p], 1) == a.H - 1;
  }
  if (!__shfl_sync(0xffffffffu, last, 0)) return;
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

// Eq. 5 and 6 of one (problem, head) vector by a CTA or a cluster, in two sweeps over memory: the sum of squared
// deviations from 1/n (the pooled vector sums to 1, so 1/n is its mean; summing deviations instead of
// squares keeps near-uniform attention from cancelling) and the mass of the floor(n / 10) largest entries.
// Counting sweeps locate the k-th largest value to 22 bits (all entries are >= 0: the order of the bit
// patterns is theirs):
//   sweep 1: histogram of bits 30..20 (exponent + 3 mantissa bits); sum of squared deviations
//   sweep 2: exact sum of the entries above the threshold bin and a histogram of bits 19..9 inside it
// The entries inside the threshold bin are then summed as count x bin midpoint: bins of the second
// level are 2^-14 wide relative to their value, far inside the metric's tolerance.
//
// A sweep's cost is its instructions: counts are predicated (a branch around each took three times as many), what lies beyond a
// vector's end is skipped, one warp walks the bins, and one CTA with an SM to itself keeps up to 16384 entries in its
// registers between the sweeps.  us without / with, chained launches over 32 heads: one layer of 16384 keys 9.0 / 7.6, of 32768
// 11.6 / 9.6, of 262144 20.2 / 17.2; 32 layers of 5003 keys 15.6 / 14.4, of 32768 58 / 50, of 131072 215 / 196.
//
// Bound by latency up to some 100 vectors, then by the shared-memory atomics and, where the vectors exceed
// L2 together, by reading them twice (1024 vectors of 131072 keys: 2 x 537 MB, 164 of 196 us).  One histogram,
// without copies for the lanes: same-address hits cost less than clearing and summing copies, whether the
// values concentrate or not (1024 vectors of 5003 / 32768 keys, before counts were predicated: 41 / 85 us with four, 20 / 59 with
// one, both with three CTAs of 512 an SM).
//
// Few long vectors are dealt out over clusters of CL CTAs, which count their own entries; the histograms are
// read through distributed shared memory, and the first CTA adds up.  A CTA takes 0.15 us per 1000 keys, mostly
// its histogram's atomics; the cluster's barriers and remote reads come to 3 us.
//
// The bits of a vector's sums must depend neither on how many threads and CTAs work on it nor on its alignment:
// entry j belongs to accumulator j mod 1024 ROWS, where ROWS follows from the length alone.  Rows of 1024 are
// dealt out to the CTAs in turn, and a thread has kAccs of the accumulators.
constexpr int kSwBins = 2048;
constexpr int kLongRows = 8;                               // ROWS of a long vector; a short one has a single row
constexpr int kLongFrom = 32768;                           // keys a short vector has at most
struct SweepShared {
  alignas(16) unsigned hist[2][kSwBins];
  float red[2][kLongRows][32], red_bin[32];                // sums of the warps, row by row
  unsigned scan[2][32], bin, rem;                          // [level] sums of the warps, or of 64 bins each
};
template <int T, int CL, int ROWS> constexpr int kAccs = ROWS == 1 ? 1024 / T : ROWS * 1024 / (T * CL);
// Applies f(entry, accumulator, whether there is one) to this CTA's entries of a[0 .. n) once each, 48 or 64 KB of loads in
// flight on an SM.
template <int T, int CL, int ROWS, class F>
__device__ __forceinline__ void sweep_from_memory(const float* __restrict__ a, int n, int rank, F f) {
  constexpr int kAt = T == 1024 ? 16 : 8, kStep = ROWS == 1 ? T : T * CL, kMine = kAccs<T, CL, ROWS>;
  constexpr int kChunk = kMine > kAt ? kMine : kAt;
  if (ROWS == 1 && rank > 0) return;
  int first = rank * T;
  float v[kAt];
  for (; first + (kChunk - 1) * kStep + T <= n; first += kChunk * kStep) {
#pragma unroll
    for (int h = 0; h < kChunk; h += kAt) {
#pragma unroll
      for (int u = 0; u < kAt; ++u) v[u] = a[first + threadIdx.x + (h + u) * kStep];
#pragma unroll
      for (int u = 0; u < kAt; ++u) f(v[u], (h + u) & (kMine - 1), true);
    }
  }
  const int j = first + threadIdx.x;
#pragma unroll
  for (int h = 0; h < kChunk; h += kAt) {
    if (first + h * kStep >= n) return;
#pragma unroll
    for (int u = 0; u < kAt; ++u) v[u] = j + (h + u) * kStep < n ? a[j + (h + u) * kStep] : 0.f;
#pragma unroll
    for (int u = 0; u < kAt; ++u)
      if (first + (h + u) * kStep < n) f(v[u], (h + u) & (kMine - 1), j + (h + u) * kStep < n);
  }
}
// Sums of N accumulators (a power of two) over each warp, to the rows they belong to.  While there are several, a
// lane hands half of them to its partner and keeps the other half: 16 shuffles for 16 sums instead of 80
// (1024 vectors of 131072 keys 210 us, now 208), and the same bits.
template <int T, int CL, int N>
__device__ __forceinline__ void warp_sums(float (&v)[N], float* red, int rank) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int o = 16;
#pragma unroll
  for (int n = N / 2; n > 0; n /= 2, o /= 2) {
    const bool upper = lane & o;
#pragma unroll
    for (int i = 0; i < n; ++i) {
      const float other = __shfl_xor_sync(0xffffffffu, upper ? v[i] : v[i + n], o);
      v[i] = (upper ? v[i + n] : v[i]) + other;
    }
  }
#pragma unroll
  for (; o > 0; o /= 2) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
  const int k = lane / (32 / N);                           // the sum this lane ended up with
  if (lane % (32 / N) == 0) red[T == 1024 ? (k * CL + rank) * 32 + warp : k * (T / 32) + warp] = v[0];
}
// `p` in CTA `rank` of the cluster.
template <int CL, class P>
__device__ __forceinline__ P* in_cta(P* p, int rank) {
  return CL > 1 ? cg::this_cluster().map_shared_rank(p, rank) : p;
}
template <int CL>
__device__ __forceinline__ void all_ctas() {
  if (CL > 1) cg::this_cluster().sync();
  else __syncthreads();
}
template <int CL>
__device__ __forceinline__ unsigned count_of(unsigned* bin) {
  unsigned c = 0;
#pragma unroll
  for (int r = 0; r < CL; ++r) c += *in_cta<CL>(bin, r);
  return c;
}
// Total over the rows (one warp calls, after all_ctas; fixed order, all loads in flight together).
template <int CL, int ROWS>
__device__ __forceinline__ float total_of(float (*red)[32]) {
  float s[ROWS], total = 0.f;
#pragma unroll
  for (int r = 0; r < ROWS; ++r) s[r] = in_cta<CL>(red[r], r % CL)[threadIdx.x];
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s[r] += __shfl_xor_sync(0xffffffffu, s[r], o);
    total += s[r];
  }
  return total;
}
// Lane l: the l-th of 32 counts from the top.  Where the wanted rank falls; `rest` becomes the rank inside it.
__device__ __forceinline__ int find_rank(unsigned count, unsigned& rest) {
  const int lane = threadIdx.x & 31;
  unsigned incl = count;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  const unsigned before = incl - count;
  const int at = __ffs(__ballot_sync(0xffffffffu, before < rest && rest <= incl)) - 1;
  rest -= __shfl_sync(0xffffffffu, before, at);
  return at;
}
// Once all warps have counted: walks the bins of a histogram from the top.  s.bin holds the `remaining`-th largest candidate,
// s.rem is the rank still wanted inside it.  32 groups of 64 bins first, summed by their warps, then, in one warp, the
// groups and the bins of one of them.
template <int T>
__device__ __forceinline__ void sweep_pick(SweepShared& s, int level, unsigned remaining) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint2* const pairs = reinterpret_cast<const uint2*>(s.hist[level]);
  __syncthreads();
#pragma unroll
  for (int g = warp; g < 32; g += T / 32) {
    const uint2 c = pairs[g * 32 + lane];
    const unsigned sum = __reduce_add_sync(0xffffffffu, c.x + c.y);
    if (lane == 0) s.scan[level][g] = sum;
  }
  __syncthreads();
  if (warp == 0) {
    unsigned rest = remaining;
    const int group = 31 - find_rank(s.scan[level][31 - lane], rest), pair = 32 * group + 31 - lane;
    const uint2 c = pairs[pair];
    const int at = find_rank(c.x + c.y, rest);
    if (lane == at) {
      s.bin = (unsigned)(2 * pair) + (rest <= c.y ? 1u : 0u);
      s.rem = rest <= c.y ? rest : rest - c.y;
    }
  }
  __syncthreads();
}
// The same for a cluster, in two steps of one warp: 32 groups of 64 bins, summed by their owners before the
// barrier, then the bins of one group.
template <int CL>
__device__ __forceinline__ void cluster_pick(SweepShared& s, int level, unsigned remaining) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned* const hist = s.hist[level];
  unsigned* const groups = s.scan[level];
  __syncthreads();
  const uint2 mine = reinterpret_cast<const uint2*>(hist)[warp * 32 + lane];
  const unsigned sum = __reduce_add_sync(0xffffffffu, mine.x + mine.y);
  if (lane == 0) groups[warp] = sum;
  all_ctas<CL>();
  if (warp == 0) {
    unsigned rest = remaining, lo = 0, hi = 0;
    const int group = 31 - find_rank(count_of<CL>(&groups[31 - lane]), rest);
    const int pair = 32 * group + 31 - lane;
#pragma unroll
    for (int r = 0; r < CL; ++r) {
      const uint2 c = *in_cta<CL>(reinterpret_cast<uint2*>(hist) + pair, r);
      lo += c.x;
      hi += c.y;
    }
    const int at = find_rank(lo + hi, rest);
    if (lane == at) {
      s.bin = (unsigned)(2 * pair) + (rest <= hi ? 1u : 0u);
      s.rem = rest <= hi ? rest : rest - hi;
    }
  }
  __syncthreads();
}
template <int T, int CL, int ROWS>
__device__ __forceinline__ void sweep_cta(const FinishArgs& a, SweepShared& s, const Problem& pb, int vec) {
  const int tid = threadIdx.x, rank = CL > 1 ? (int)(blockIdx.x % CL) : 0, n = pb.n;
  const float* x = pb.cols + (size_t)(vec % a.H) * a.col_stride;
  const float mean = 1.f / (float)n;
  float acc[kAccs<T, CL, ROWS>] = {};
  unsigned b1 = 0;
  auto first_sweep = [&](float v, int k, bool in) {
    const float dv = v - mean;
    acc[k] = in ? fmaf(dv, dv, acc[k]) : acc[k];
    count_if(in, &s.hist[0][(__float_as_uint(v) >> 20) & 0x7ffu]);
  };
  auto second_sweep = [&](float v, int k, bool in) {
    const unsigned u = __float_as_uint(v), top = (u >> 20) & 0x7ffu;
    acc[k] += in && top > b1 ? v : 0.f;
    count_if(in && top == b1, &s.hist[1][(u >> 9) & 0x7ffu]);
  };
  auto pick = [&](int level, unsigned remaining) {
    if (ROWS > 1 || rank == 0) warp_sums<T, CL>(acc, s.red[level][0], rank);
    if (CL > 1) cluster_pick<CL>(s, level, remaining);
    else sweep_pick<T>(s, level, remaining);
#pragma unroll
    for (float& m : acc) m = 0.f;
  };
  // One CTA with an SM to itself keeps a short vector's entries in its registers from sweep to sweep.
  constexpr int kHold = T == 1024 && CL == 1 && ROWS == 1 ? 16 : 0;
  if (kHold > 0 && n <= kHold * T) {
    constexpr int kAt = 4;
    float v[kHold > 0 ? kHold : 1];
#pragma unroll
    for (int h = 0; h < kHold; h += kAt) {
      if (h * T >= n) break;
#pragma unroll
      for (int u = h; u < h + kAt; ++u) v[u] = tid + u * T < n ? x[tid + u * T] : 0.f;
    }
    auto all = [&](auto f) {
#pragma unroll
      for (int h = 0; h < kHold; h += kAt) {
        if (h * T >= n) break;
#pragma unroll
        for (int u = h; u < h + kAt; ++u) f(v[u], 0, tid + u * T < n);
      }
    };
    all(first_sweep);
    pick(0, (unsigned)max(1, n / 10));
    b1 = s.bin;
    all(second_sweep);
  } else {
    sweep_from_memory<T, CL, ROWS>(x, n, rank, first_sweep);
    pick(0, (unsigned)max(1, n / 10));
    b1 = s.bin;
    sweep_from_memory<T, CL, ROWS>(x, n, rank, second_sweep);
  }
  const unsigned rem1 = s.rem;
  pick(1, rem1);
  const unsigned b2 = s.bin, rem2 = s.rem;
  if (rank == 0) {
    // entries of the threshold bin above sub-bin b2, and rem2 entries of sub-bin b2 itself
    constexpr int kAccsBin = 1024 / T;
    float in_bin[kAccsBin] = {};
#pragma unroll
    for (int q = 0; q < kSwBins / T; ++q) {
      const int b = q * T + tid;
      const float mid = __uint_as_float((b1 << 20) | ((unsigned)b << 9) | 0x100u);
      const unsigned cnt = (unsigned)b > b2 ? count_of<CL>(&s.hist[1][b]) : ((unsigned)b == b2 ? rem2 : 0u);
      float& to = in_bin[q & (kAccsBin - 1)];
      to = fmaf((float)cnt, mid, to);
    }
    warp_sums<T, 1>(in_bin, s.red_bin, 0);
    __syncthreads();
    if (tid < 32) {
      const float sq = total_of<CL, ROWS>(s.red[0]), mass = total_of<CL, ROWS>(s.red[1]);
      head_done(a, vec, mean, sq, mass + total_of<1, 1>(&s.red_bin));
    }
  }
  if (CL > 1) all_ctas<CL>();                              // no CTA leaves while the first one reads its memory
}
// LONG: some vector has more than kLongFrom keys.  Short ones have a kernel of their own: with both forms in one
// kernel a launch over 32 vectors of 4096 keys took a microsecond longer.
// FRONT: all statistics, then all sums: where every vector has an SM, and where there are no sums (a vector that follows
// from the block's index alone leaves the sweeps the registers for another load: 1024 vectors of 131072 keys took 219 us, 234 in
// the other order, before counts were predicated).
// Else problem after problem, its sums right behind its statistics, so that they find in L2 what these have
// read, and the last problem first: of the columns the scorer has just written L2 still holds the last ones.  (The lines between
// the two are at launch_finish.  A batch of four prompts, 128 vectors, lost 2 us a layer by it.  Clusters of four for many
// long vectors, fewer of them at a time, took 11 to 22 us more than this order for 28 layers of 65536 keys and 32 of 131072.)
template <int VEC, int T, int CL, bool LONG, bool FRONT>
__global__ void __launch_bounds__(T, T == 256 ? 6 : T == 512 ? 3 : 1) finish(const __grid_constant__ FinishArgs a) {
  __shared__ union { SweepShared stats; SumShared<VEC> sum; } sh;
  const int per = a.stat_ctas + a.chunks, at = FRONT ? 0 : blockIdx.x / per, in_front = FRONT ? a.n_prob * a.stat_ctas : a.stat_ctas;
  const int b = blockIdx.x - at * per;                     // FRONT: of the launch; else of its problem
  const bool stats = b < in_front;
  pdl_trigger();
  if (stats)
    for (int i = threadIdx.x; i < 2 * kSwBins; i += T) sh.stats.hist[0][i] = 0;
  pdl_wait();
  __syncthreads();
  if (stats) {
    const int vec = FRONT ? blockIdx.x / CL : (a.n_prob - 1 - at) * a.H + b / CL;
    const Problem pb = problem_of(a, vec / a.H);
    if (LONG && pb.n > kLongFrom) sweep_cta<T, CL, kLongRows>(a, sh.stats, pb, vec);
    else sweep_cta<T, CL, 1>(a, sh.stats, pb, vec);
  } else {
    const int c = b - in_front, p = FRONT ? c / a.chunks : a.n_prob - 1 - at;
    if (p < a.n_prob) sum_block<VEC, T>(a, sh.sum, p, FRONT ? c - p * a.chunks : c);   // the grid is whole clusters
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

// Eq. 7-9, then the same recursion.  Every block finds the pivot for itself, so that no launch and no host round trip comes
// between the metrics and the centrality, while its first kEarly layers are on their way.  The last block sums nothing: it
// tells the host, beside the others' sums, in words that carry the call's tag, so that none waits for another.
// Bound by latency, above all by fetching instructions that nothing has run before: with one warp for the three columns
// and four rounds of layers, all unrolled, a dozen double divisions written out, the smallest launches took 8.8 to 10 us by
// themselves; with a warp per column and rolled loops 5.2 to 5.4 (whole prefills 3.5 to 4.3 us less).
constexpr int kPivotThreads = 128, kEarly = 8;
template <int VEC>
__global__ void __launch_bounds__(kPivotThreads)
accumulate_at_pivot(const float* __restrict__ s_hist, long long row_stride, int n_layers, int n, float lambda,
                    const float* __restrict__ metrics, float3 weights, int l_limit, float* __restrict__ c_out,
                    volatile unsigned long long* host, unsigned tag) {
  using T = typename Keys<VEC>::T;
  __shared__ float m_s[3 * kMaxStatLayers];
  __shared__ double t_s[3][kMaxStatLayers];
  __shared__ int pivot_s;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool tells = blockIdx.x == gridDim.x - 1;
  const int j = (blockIdx.x * kPivotThreads + tid) * VEC;
  const bool sums = !tells && j < n;
  pdl_trigger();
  pdl_wait();
  for (int i = tid; i < 3 * n_layers; i += kPivotThreads) m_s[i] = metrics[i];
  T early[kEarly] = {};
  if (sums) {
#pragma unroll
    for (int l = 0; l < kEarly; ++l)
      if (l < n_layers) early[l] = *reinterpret_cast<const T*>(s_hist + (size_t)l * row_stride + j);
  }
  __syncthreads();
  if (warp < 3) {                                          // a column each
    const double w = warp == 0 ? weights.x : warp == 1 ? weights.y : weights.z;
    auto step = [&](int l) {                               // Eq. 8 takes the gradient of -entropy
      const double d = (double)m_s[3 * l + warp] - (double)m_s[3 * l - 3 + warp];
      return warp == 0 ? -d : d;
    };
    double lo = INFINITY, hi = -INFINITY;
    int nan = 0;
#pragma unroll 1
    for (int l = lane; l < n_layers; l += 32) {
      nan |= isnan(m_s[3 * l + warp]);
      if (l == 0) continue;
      const double d = step(l);
      lo = d < lo ? d : lo;
      hi = d > hi ? d : hi;
    }
#pragma unroll 1
    for (int o = 16; o > 0; o >>= 1) {
      const double a = __shfl_xor_sync(0xffffffffu, lo, o), b = __shfl_xor_sync(0xffffffffu, hi, o);
      lo = a < lo ? a : lo;
      hi = b > hi ? b : hi;
    }
    const bool usable = !__any_sync(0xffffffffu, nan) && hi > lo;
#pragma unroll 1
    for (int l = lane; l < n_layers; l += 32)
      t_s[warp][l] = usable && l > 0 ? __ddiv_rn(__dmul_rn(w, __dsub_rn(step(l), lo)), __dsub_rn(hi, lo)) : 0.0;
  }
  __syncthreads();
  if (warp == 0) {
    double best = -INFINITY;
    int at = kMaxStatLayers;
#pragma unroll 1
    for (int l = lane; l < n_layers; l += 32) {
      const double t = __dadd_rn(__dadd_rn(t_s[0][l], t_s[1][l]), t_s[2][l]);
      if (l > 0 && t > best) { best = t; at = l; }
      if (tells) host[1 + l] = (unsigned long long)tag << 32 | (unsigned)__float_as_int((float)t);
    }
#pragma unroll 1
    for (int o = 16; o > 0; o >>= 1) {
      const double b = __shfl_xor_sync(0xffffffffu, best, o);
      const int i = __shfl_xor_sync(0xffffffffu, at, o);
      if (b > best || (b == best && i < at)) { best = b; at = i; }
    }
    if (at == kMaxStatLayers) at = n_layers >= 2 ? 1 : 0;   // one layer, or nothing compares
    if (n_layers >= 2 && l_limit >= 0 && at > l_limit) at = l_limit;
    if (lane == 0) {
      pivot_s = at;
      if (tells) host[0] = (unsigned long long)tag << 32 | (unsigned)at;
    }
  }
  if (tells) return;
  __syncthreads();
  if (!sums) return;
  const int pivot = pivot_s;
  T c{};
#pragma unroll
  for (int l = 0; l < kEarly; ++l)
    if (l <= pivot) c = decay(lambda, c, early[l]);
#pragma unroll 8
  for (int l = kEarly; l <= pivot; ++l) c = decay(lambda, c, *reinterpret_cast<const T*>(s_hist + (size_t)l * row_stride + j));
  *reinterpret_cast<T*>(c_out + j) = c;
}

}  // namespace

constexpr int kNarrowMany = 8192;    // keys up to which six CTAs of 256 are the better ones for many vectors, sums or not

template <int VEC>
static cudaError_t launch_finish(FinishArgs& a, int longest, int sms, cudaStream_t st) {
  a.chunks = a.row_ent ? (longest + kSumLanes * VEC - 1) / (kSumLanes * VEC) : 0;
  const int sums = a.n_prob * a.chunks;
  if (!a.with_stats) return launch_pdl(sum_layers<VEC>, dim3(sums), dim3(kSumThreads), 0, st, a);
  // An SM per vector: as many threads as a CTA can have.  More vectors than SMs: several CTAs an SM fill each
  // other's gaps between barriers, six of 256 for short vectors, three of 512 for long ones.  us, three of 512 / six of 256:
  // statistics alone of 32 layers of 32 heads, 1500 keys 14.1 / 10.6, 5003 18.3 / 14.9, 8192 19.7 / 18.0, 16384 27.9 /
  // 28.3, 32768 56 / 70; of 10 layers, which three of 512 take in one go, 5003 keys 8.5 / 10.1, 8192 9.0 / 11.8; whole prefills of
  // 32 layers, 1500 keys 150.0 / 144.7, 5003 298.8 / 288.6, 8192 428.6 / 424.5, of 14 layers of 5003 keys 143.9 / 141.3, of 10 121.6
  // / 123.9.
  // Few long vectors: clusters, as large as leaves room for all of them at once.
  const int n_vec = a.n_prob * a.H, room = longest > kLongFrom ? sms * 7 / 8 / n_vec : 1;
  const int cl = 8 * n_vec <= sms * 3 / 4 && room >= 8 ? 8 : room >= 4 ? 4 : room >= 2 ? 2 : 1;
  a.stat_ctas = a.H * cl;
  const dim3 grid((n_vec * cl + sums + cl - 1) / cl * cl), wide(1024), narrow(512);
  if (cl == 8) return launch_cluster<8>(finish<VEC, 1024, 8, true, true>, grid, wide, 0, st, a);
  if (cl == 4) return launch_cluster<4>(finish<VEC, 1024, 4, true, true>, grid, wide, 0, st, a);
  if (cl == 2) return launch_cluster<2>(finish<VEC, 1024, 2, true, true>, grid, wide, 0, st, a);
  if (n_vec <= sms)
    return longest > kLongFrom ? launch_pdl(finish<VEC, 1024, 1, true, true>, grid, wide, 0, st, a)
                               : launch_pdl(finish<VEC, 1024, 1, false, true>, grid, wide, 0, st, a);
  // Sums behind their statistics only where the statistics take several goes of three CTAs an SM.  Whole prefills, 32 heads, us
  // in front / behind: 1500 keys, 6 layers 74.6 / 77.6, 14 layers 86.5 / 83.5; 5003 keys, 6 layers 97.6 / 100.5, 10 122.4 /
  // 124.4, 14 141.4 / 141.0; 20000 keys, 10 layers 333 / 339; 24 of 32768 1315 / 1288; 65536 keys, 14 layers 1492 / 1465, 20 2125 /
  // 2053, 24 2516 / 2478.  No more apart than the runs of one: 20 and 32 layers of 5003, 14 to 24 of 8193, 20 to 28 of 20000, 20
  // and 32 of 32768, 20 and 24 of 131072.
  const bool several = n_vec > (longest > kNarrowMany ? 5 : 3) * sms;
  if (!sums || !several)
    return longest > kLongFrom ? launch_pdl(finish<VEC, 512, 1, true, true>, grid, narrow, 0, st, a)
           : longest > kNarrowMany || n_vec <= 3 * sms ? launch_pdl(finish<VEC, 512, 1, false, true>, grid, narrow, 0, st, a)
                                                        : launch_pdl(finish<VEC, 256, 1, false, true>, grid, dim3(256), 0, st, a);
  return longest > kLongFrom ? launch_pdl(finish<VEC, 512, 1, true, false>, grid, narrow, 0, st, a)
                             : launch_pdl(finish<VEC, 256, 1, false, false>, grid, dim3(256), 0, st, a);
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

cudaError_t launch_head_stats_batch(const Ctx& ctx, const float* cols, long long layer_stride, long long col_stride,
                                    int n_layers, int n, float* metrics, cudaStream_t st) {
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
                                       const float* metrics, const float* weights, int l_limit, float* c_out,
                                       unsigned long long* host, unsigned tag, cudaStream_t st) {
  const float3 w = make_float3(weights[0], weights[1], weights[2]);
  const auto blocks = [](int threads) { return dim3((threads + kPivotThreads - 1) / kPivotThreads + 1); };
  if (n % 4 == 0 && row_stride % 4 == 0 && (uintptr_t)s_hist % 16 == 0 && (uintptr_t)c_out % 16 == 0)
    return launch_pdl(accumulate_at_pivot<4>, blocks(n / 4), dim3(kPivotThreads), 0, st, s_hist, row_stride, n_layers, n, lambda,
                      metrics, w, l_limit, c_out, (volatile unsigned long long*)host, tag);
  return launch_pdl(accumulate_at_pivot<1>, blocks(n), dim3(kPivotThreads), 0, st, s_hist, row_stride, n_layers, n, lambda, metrics,
                    w, l_limit, c_out, (volatile unsigned long long*)host, tag);
}

}  // namespace skv
