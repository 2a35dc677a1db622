// Budgeted token selection (top-k of the prefix, ties to the lower index, output in position
// order, window appended), exact: three levels of 11, 11 and 10 bits find the k-th largest key (radix.cuh), then every
// kept token's place in the output follows from ballots and one scan of the warps' counts (a warp's tokens are
// consecutive).  A cluster of CL CTAs shares one vector, each CTA a contiguous slice that it
// holds in registers (up to ITEMS tokens a thread; a longer slice is read again per level).
//
// Bound by the chain of barriers, not by memory; with several tokens a thread, by the instructions for each: one vector
// of 131072 tokens took 18.7 us, 5.8 of them for the output's places, scanned per (group of 1024 tokens, warp) with equal
// keys counted whether there are any or not; now 12.5 and 3.
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

// Two CTAs an SM for the many short vectors that need them.  Clusters of up to eight items a thread have an SM per CTA: bound
// to 32 registers they spilled (8 / 16 vectors of 32768 tokens 13.0 / 14.8 us instead of 11.2 / 11.3).
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
  const bool own = !a.packed && vec == a.batch;      // the extra vector
  const float* x = own ? a.extra.scores : a.scores + (a.packed ? (size_t)a.cu[vec] : (size_t)vec * a.row_stride);
  const int n = a.packed ? a.cu[vec + 1] - a.cu[vec] : a.n, budget = own ? a.extra.budget : a.packed ? a.budgets[vec] : a.budget;
  int* out = own ? a.extra.idx_out : a.out + (size_t)vec * a.out_stride;
  const int prefix_len = n - a.window, k = budget - a.window;
  cluster_barrier<CL>();                             // all CTAs of the cluster run before any remote access
  pdl_wait();
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
  int n_mine = 0;                                    // this thread's tokens of the loaded chunk
  // a warp's tokens are consecutive; item e of this thread: first + 32 e
  auto first_of = [&](int c) { return lo + c * kChunk + warp * (32 * ITEMS) + lane; };
  auto load = [&](int c) {
    const int first = first_of(c);
    n_mine = min(ITEMS, (hi - first + 31) >> 5);     // (none where this is not positive)
    float v[ITEMS];
#pragma unroll
    for (int e = 0; e < ITEMS; ++e) v[e] = e < n_mine ? x[first + 32 * e] : 0.f;
#pragma unroll
    for (int e = 0; e < ITEMS; ++e) key[e] = order_key(v[e]);
  };

  if (chunks == 1) load(0);
  // kept: every key > above, and the first need_eq of the keys equal to thr.  (Keys start at 0x007fffff, minus infinity, so that
  // thr - 1 does not wrap.  They end at 0xffffffff, a NaN: where that is the threshold, nothing is above it.)
  unsigned above = 0, thr = 0, need_eq = 0;
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
          radix_count(s, level, radix_digit(key[e], level), e < n_mine && (key[e] & mask) == thr);
      }
      unsigned digit, in;
      radix_pick(s, level, remaining, digit, in);
      thr |= digit << radix_shift(level);
      if (in == remaining) break;                    // all keys of the digit are kept: no need to look inside
    }
    above = level < kRxLevels ? thr - 1 : thr;
    need_eq = level < kRxLevels ? 0 : remaining;
  }

  // Place of a token in the output = (#kept outright before it) + min(#equal before it, need_eq).  Counts of this warp in the
  // loaded chunk:
  unsigned w_gt = 0, w_eq = 0;
  auto tally = [&]() {
    w_gt = w_eq = 0;
#pragma unroll
    for (int e = 0; e < ITEMS; ++e) w_gt += __popc(__ballot_sync(0xffffffffu, e < n_mine && key[e] > above));
    if (need_eq == 0) return;                        // keys that differ: what stays is above
#pragma unroll
    for (int e = 0; e < ITEMS; ++e) w_eq += __popc(__ballot_sync(0xffffffffu, e < n_mine && key[e] == thr));
  };
  auto leave = [&](unsigned gt, unsigned eq) {
    if (lane == 0) { s.scratch[0][warp] = gt; s.scratch[1][warp] = eq; }
    __syncthreads();
  };
  unsigned gt_run = 0, eq_run = 0;                   // before this CTA's slice, then before the chunk
  if (CL > 1) {
    unsigned all_gt = 0, all_eq = 0;
    for (int c = 0; c < chunks; ++c) {
      if (chunks > 1) load(c);
      tally();
      all_gt += w_gt;
      all_eq += w_eq;
    }
    leave(all_gt, all_eq);
    if (warp < 2) {
      const unsigned t = __reduce_add_sync(0xffffffffu, s.scratch[warp][lane]);
      if (lane < CL) cg::this_cluster().map_shared_rank(&cta_tot[0][0], lane)[warp * CL + rank] = t;
    }
    cluster_barrier<CL>();
    for (int r = 0; r < rank; ++r) { gt_run += cta_tot[0][r]; eq_run += cta_tot[1][r]; }
  }
  const unsigned below = (1u << lane) - 1u;
  for (int c = 0; c < chunks; ++c) {
    if (chunks > 1) {
      load(c);
      __syncthreads();                               // the counts of the chunk before have been read
    }
    if (CL == 1 || chunks > 1) {                     // else they are there
      tally();
      leave(w_gt, w_eq);
    }
    const unsigned g = s.scratch[0][lane], g_incl = warp_scan(g, lane);
    unsigned gt_at = gt_run + __shfl_sync(0xffffffffu, g_incl - g, warp), eq_at = 0;
    gt_run += __shfl_sync(0xffffffffu, g_incl, 31);
    if (need_eq) {
      const unsigned q = s.scratch[1][lane], q_incl = warp_scan(q, lane);
      eq_at = eq_run + __shfl_sync(0xffffffffu, q_incl - q, warp);
      eq_run += __shfl_sync(0xffffffffu, q_incl, 31);
    }
    const int first = first_of(c);
    if (need_eq == 0) {
#pragma unroll
      for (int e = 0; e < ITEMS; ++e) {
        const bool gt = e < n_mine && key[e] > above;
        const unsigned bg = __ballot_sync(0xffffffffu, gt);
        if (gt) out[gt_at + __popc(bg & below)] = first + 32 * e;
        gt_at += __popc(bg);
      }
    } else {
#pragma unroll
      for (int e = 0; e < ITEMS; ++e) {
        const bool in = e < n_mine, gt = in && key[e] > above, eq = in && key[e] == thr;
        const unsigned bg = __ballot_sync(0xffffffffu, gt), be = __ballot_sync(0xffffffffu, eq);
        const unsigned eq_before = eq_at + __popc(be & below);
        if (gt || (eq && eq_before < need_eq)) out[gt_at + __popc(bg & below) + min(eq_before, need_eq)] = first + 32 * e;
        gt_at += __popc(bg);
        eq_at += __popc(be);
      }
    }
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

// One CTA while that is a matter of three barriers a level; beyond, as many CTAs with as few items each as leave all
// vectors running at once (a CTA has an SM, clusters do not cross a GPC: 148 SMs run 15 clusters of eight or 33 of four, and the
// lines are theirs).  us, CTAs x items, for 1 / 8 / 33 vectors, chained launches (of which some take 1.2 to 2 us more
// than others with the same work): 1777 tokens 1 x 4 4.9 / 4.0 / 4.5, 2 x 2 5.4 / 5.5 / 5.5; 8192 1 x 8 5.1 / 5.2 / 6.4, 4 x 2 5.7 /
// 5.9 / 7.2; 16384 4 x 4 7.8 / 6.4 / 8.0, 1 x 16 8.9 / 7.5 / 9.1, 8 x 2 7.7 / 6.5 / 18.9; 32768 8 x 4 6.6 / 8.5 / 22.2, 4 x 8
// 7.2 / 9.2 / 9.3, 2 x 16 9.2 / 11.3 / 11.4; 65536 8 x 8 9.6 / 10.0 / 25.6, 4 x 16 11.3 / 11.4 / 11.8; 131072 8 x 16 12.5 /
// 12.8 / 33.6, 4 x 32 15.9 / 16.1 / 19.8.  15 / 16 vectors by eight, by four: 32768 tokens 8.8 / 13.5, 9.0 / 9.0; 65536 10.1 /
// 15.5, 11.4 / 11.4; 131072 12.5 / 19.7, 16.3 / 16.3.
// Where eight CTAs hold a vector in registers and four would read it again for every digit, two goes of eight are still the
// faster ones: 200000 tokens, 16 / 30 / 31 vectors 30 / 33 / 44, by four 41; 262144 31 / 34 / 42, by four 43.  Where both
// read again they are not: 400000 tokens, 15 / 16 / 30 vectors 42 / 75 / 83, by four 75.
cudaError_t dispatch(const SelectArgs& a, int longest, cudaStream_t st) {
  if (longest <= 4 * kRxThreads) return launch<1, 4>(a, st);
  if (longest <= 8 * kRxThreads) return launch<1, 8>(a, st);
  const int vectors = a.batch + (a.extra.scores ? 1 : 0);
  const bool again = longest > 4 * 32 * kRxThreads && longest <= 8 * 32 * kRxThreads;
  const bool by_eight = vectors <= (again ? 30 : 15), by_four = vectors <= 33;
  if (longest <= 16 * kRxThreads) return by_four ? launch<4, 4>(a, st) : launch<1, 16>(a, st);
  if (longest <= 32 * kRxThreads) return by_eight ? launch<8, 4>(a, st) : by_four ? launch<4, 8>(a, st) : launch<2, 16>(a, st);
  if (longest <= 64 * kRxThreads) return by_eight ? launch<8, 8>(a, st) : launch<4, 16>(a, st);
  if (!by_eight) return launch<4, 32>(a, st);
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
