// Budgeted token selection (top-k of the prefix, ties to the lower index, output in position
// order, window appended), exact: three levels of 11, 11 and 10 bits find the k-th largest key (radix.cuh), then every
// kept token's place in the output follows from ballots and one scan of the counts per (group of
// 1024 tokens, warp).  A cluster of CL CTAs shares one vector, each CTA a contiguous slice that it
// holds in registers (up to ITEMS tokens a thread; a longer slice is read again per level).
//
// Bound by the chain of barriers, not by memory.
#include <atomic>

#include "radix.cuh"

namespace skv {
namespace {

struct SelectArgs {
  const float* scores;
  int* out;
  long long row_stride, out_stride;    // between the vectors of a uniform call; rows of `out`
  int n, budget, window, batch;
  // packed sequences: vector b is scores[cu[b] .. cu[b + 1]) with its own budget; the row's remainder reads -1
  int packed;
  int cu[kMaxBatch + 1], budgets[kMaxBatch];
  SelectExtra extra;                   // vector `batch` of a uniform call, if it has scores
};

// Two CTAs an SM for the many short vectors that need them.  Clusters of up to eight items a thread serve at most 17 vectors,
// 68 CTAs: bound to 32 registers they spilled (8 / 16 vectors of 32768 tokens 13.0 / 14.8 us, now 11.2 / 11.3; of 12000
// 8.1 / 8.3, now 7.7 / 7.7).
template <int CL, int ITEMS>
__global__ void __launch_bounds__(kRxThreads, CL == 1 && ITEMS <= 8 ? 2 : 1) select_topk(const __grid_constant__ SelectArgs a) {
  extern __shared__ __align__(16) unsigned char sel_smem[];
  RadixShared<CL>& s = *reinterpret_cast<RadixShared<CL>*>(sel_smem);
  __shared__ unsigned cta_tot[2][CL];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = CL > 1 ? (int)cg::this_cluster().block_rank() : 0;
  const int vec = blockIdx.x / CL;
  pdl_trigger();
  radix_clear(s);
  cluster_barrier<CL>();                             // all CTAs of the cluster run before any remote access
  pdl_wait();
  const bool own = !a.packed && vec == a.batch;      // the extra vector
  const float* x = own ? a.extra.scores : a.scores + (a.packed ? (size_t)a.cu[vec] : (size_t)vec * a.row_stride);
  const int n = a.packed ? a.cu[vec + 1] - a.cu[vec] : a.n, budget = own ? a.extra.budget : a.packed ? a.budgets[vec] : a.budget;
  int* out = own ? a.extra.idx_out : a.out + (size_t)vec * a.out_stride;
  const int prefix_len = n - a.window, k = budget - a.window;
  if (rank == 0) {
    for (int i = tid; i < a.window; i += kRxThreads) out[k + i] = prefix_len + i;
    if (a.packed)
      for (long long i = budget + tid; i < a.out_stride; i += kRxThreads) out[i] = -1;
  }
  if (k <= 0) return;                                // the same decision in every CTA of the cluster

  const int per = (prefix_len + CL - 1) / CL;
  const int lo = min(prefix_len, rank * per), hi = min(prefix_len, lo + per);
  constexpr int kChunk = kRxThreads * ITEMS;
  const int chunks = (per + kChunk - 1) / kChunk;    // more than one: the slice does not fit the registers
  unsigned key[ITEMS];
  // token of item e: base + e * 1024 + tid
  auto load = [&](int c) {
    const int base = lo + c * kChunk;
    float v[ITEMS];
#pragma unroll
    for (int e = 0; e < ITEMS; ++e) {
      const int j = base + e * kRxThreads + tid;
      v[e] = j < hi ? x[j] : 0.f;
    }
#pragma unroll
    for (int e = 0; e < ITEMS; ++e) key[e] = order_key(v[e]);
  };
  auto valid = [&](int c, int e) { return lo + c * kChunk + e * kRxThreads + tid < hi; };

  if (chunks == 1) load(0);
  // kept: every key >= ge, and the first need_eq of the keys equal to thr
  unsigned ge = 0, thr = 0, need_eq = 0;
  if (k < prefix_len) {
    unsigned remaining = (unsigned)k;
    int level = 0;
#pragma unroll 1
    for (; level < kRxLevels; ++level) {
      const unsigned mask = level == 0 ? 0u : 0xffffffffu << radix_shift(level - 1);
      for (int c = 0; c < chunks; ++c) {
        if (chunks > 1) load(c);
#pragma unroll
        for (int e = 0; e < ITEMS; ++e)
          if (valid(c, e) && (key[e] & mask) == thr) radix_count(s, level, radix_digit(key[e], level));
      }
      unsigned digit, in;
      radix_pick(s, level, remaining, digit, in);
      thr |= digit << radix_shift(level);
      if (in == remaining) break;                    // all keys of the digit are kept: no need to look inside
    }
    ge = level < kRxLevels ? thr : thr + 1;
    need_eq = level < kRxLevels ? 0 : remaining;
  }

  // keys kept outright / equal to the threshold in this CTA's slice -> where the slice starts
  unsigned gt_run = 0, eq_run = 0;
  if (CL > 1) {
    unsigned my_gt = 0, my_eq = 0;
    for (int c = 0; c < chunks; ++c) {
      if (chunks > 1) load(c);
#pragma unroll
      for (int e = 0; e < ITEMS; ++e) {
        my_gt += valid(c, e) && key[e] >= ge ? 1u : 0u;
        my_eq += valid(c, e) && key[e] < ge && key[e] == thr ? 1u : 0u;
      }
    }
    my_gt = __reduce_add_sync(0xffffffffu, my_gt);
    my_eq = __reduce_add_sync(0xffffffffu, my_eq);
    if (lane == 0) { s.scratch[warp] = my_gt; s.scratch[32 + warp] = my_eq; }
    __syncthreads();
    if (warp < 2) {
      const unsigned t = __reduce_add_sync(0xffffffffu, s.scratch[warp * 32 + lane]);
      if (lane < CL) cg::this_cluster().map_shared_rank(&cta_tot[0][0], lane)[warp * CL + rank] = t;
    }
    cluster_barrier<CL>();
    for (int r = 0; r < rank; ++r) { gt_run += cta_tot[0][r]; eq_run += cta_tot[1][r]; }
  }

  // Place of token j in the output = (#kept outright before j) + min(#equal before j, need_eq).
  unsigned* const cnt = s.scratch;                   // [ITEMS][32 warps] (#outright << 16) | #equal, then exclusive sums
  unsigned* const tot = s.scratch + kRxThreads;      // [ITEMS]
  const unsigned below = (1u << lane) - 1u;
  for (int c = 0; c < chunks; ++c) {
    if (chunks > 1) load(c);
    __syncthreads();                                 // scratch is free
#pragma unroll
    for (int e = 0; e < ITEMS; ++e) {
      const bool in = valid(c, e), gt = in && key[e] >= ge, eq = in && !gt && key[e] == thr;
      const unsigned bg = __ballot_sync(0xffffffffu, gt), be = __ballot_sync(0xffffffffu, eq);
      if (lane == 0) cnt[e * 32 + warp] = (unsigned)__popc(bg) << 16 | (unsigned)__popc(be);
    }
    __syncthreads();
    if (tid < ITEMS * 32) {                          // warp e scans the warps of item e
      const unsigned v = cnt[tid];
      unsigned incl = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
      }
      cnt[tid] = incl - v;
      if (lane == 31) tot[warp] = incl;
    }
    __syncthreads();
    unsigned t_incl = lane < ITEMS ? tot[lane] : 0u;
    const unsigned t_own = t_incl;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned t = __shfl_up_sync(0xffffffffu, t_incl, o);
      if (lane >= o) t_incl += t;
    }
#pragma unroll
    for (int e = 0; e < ITEMS; ++e) {
      const bool in = valid(c, e), gt = in && key[e] >= ge, eq = in && !gt && key[e] == thr;
      const unsigned bg = __ballot_sync(0xffffffffu, gt), be = __ballot_sync(0xffffffffu, eq);
      const unsigned before = __shfl_sync(0xffffffffu, t_incl - t_own, e) + cnt[e * 32 + warp];
      const unsigned gt_before = gt_run + (before >> 16) + __popc(bg & below);
      const unsigned eq_before = eq_run + (before & 0xffffu) + __popc(be & below);
      if (gt || (eq && eq_before < need_eq))
        out[gt_before + min(eq_before, need_eq)] = lo + c * kChunk + e * kRxThreads + tid;
    }
    const unsigned all = __shfl_sync(0xffffffffu, t_incl, 31);
    gt_run += all >> 16;
    eq_run += all & 0xffffu;
  }
}

template <int CL, int ITEMS>
cudaError_t launch(const SelectArgs& a, cudaStream_t st) {
  static std::atomic<unsigned long long> ready{0};        // devices whose shared-memory limit has been raised
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (dev & 63);
  if (!(ready.load(std::memory_order_acquire) & bit)) {
    e = cudaFuncSetAttribute(select_topk<CL, ITEMS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(RadixShared<CL>));
    if (e != cudaSuccess) return e;
    ready.fetch_or(bit, std::memory_order_release);
  }
  return launch_cluster<CL>(select_topk<CL, ITEMS>, dim3((a.batch + (a.extra.scores ? 1 : 0)) * CL), dim3(kRxThreads),
                            sizeof(RadixShared<CL>), st, a);
}

// One CTA while that is a matter of three barriers a level; beyond, few vectors get more CTAs with fewer items each, and
// many (whose CTAs would not run side by side) the smallest cluster that holds one.  us for 1 / 8 / 33 vectors, chained
// launches: 1777 tokens 5.1 / 5.2 / 5.6 with 1 x 4 items (a cluster of two 6.9 / 7.0 / 7.2), 8192 7.0 / 7.2 / 8.4 with
// 1 x 8 (2 x 4: 7.2 / 7.3 / 9.0), 16384 9.9 / 10.0 / 11.7 with 1 x 16 and 7.7 / 7.8 with 4 x 4, 32768 12.0 / 12.2 /
// 14.1 with 2 x 16 and 9.3 / 11.2 with 4 x 8, 65536 13.1 / 13.3 / 16.2 with 4 x 16 and 12.5 /
// 13.2 / 26.0 with 8 x 8, 131072 18.6 with 8 x 16 and 24.1 for 33 with 4 x 32.
cudaError_t dispatch(const SelectArgs& a, int longest, cudaStream_t st) {
  if (longest <= 4 * kRxThreads) return launch<1, 4>(a, st);
  if (longest <= 8 * kRxThreads) return launch<1, 8>(a, st);
  const bool room = a.batch <= 16;                   // up to eight CTAs a vector, one per SM
  if (longest <= 16 * kRxThreads) return room ? launch<4, 4>(a, st) : launch<1, 16>(a, st);
  if (longest <= 32 * kRxThreads) return room ? launch<4, 8>(a, st) : launch<2, 16>(a, st);
  if (longest <= 64 * kRxThreads) return launch<4, 16>(a, st);
  if (!room) return launch<4, 32>(a, st);
  if (longest <= 128 * kRxThreads) return launch<8, 16>(a, st);
  return launch<8, 32>(a, st);                       // beyond 262144 tokens the slices are read again per level
}

}  // namespace

cudaError_t launch_select(const float* scores, long long row_stride, int batch, int n, int budget, int window,
                          int* idx_out, cudaStream_t st, const SelectExtra* extra) {
  SelectArgs a;
  a.extra = extra ? *extra : SelectExtra{nullptr, 0, nullptr};
  a.scores = scores; a.out = idx_out; a.row_stride = row_stride; a.out_stride = budget;
  a.n = n; a.budget = budget; a.window = window; a.batch = batch; a.packed = 0;
  return dispatch(a, n - window, st);
}

cudaError_t launch_select_packed(const float* scores, const int* cu_seqlens, const int* budgets, int batch, int window,
                                 int* idx_out, long long idx_stride, cudaStream_t st) {
  SelectArgs a;
  a.extra = SelectExtra{nullptr, 0, nullptr};
  a.scores = scores; a.out = idx_out; a.row_stride = 0; a.out_stride = idx_stride;
  a.n = a.budget = 0; a.window = window; a.batch = batch; a.packed = 1;
  int longest = 0;
  a.cu[0] = cu_seqlens[0];
  for (int b = 0; b < batch; ++b) {
    a.cu[b + 1] = cu_seqlens[b + 1];
    a.budgets[b] = budgets[b];
    longest = cu_seqlens[b + 1] - cu_seqlens[b] - window > longest ? cu_seqlens[b + 1] - cu_seqlens[b] - window : longest;
  }
  return dispatch(a, longest, st);
}

}  // namespace skv
