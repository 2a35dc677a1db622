// Tensor-core scorer of ONE layer of few keys (or a packed batch of one sequence), wide windows: what a streamed prompt's
// layers and those past the pivot call once a layer, where latency counts.
//
// The arithmetic is that of score_tc.cuh's wide layout, to the bit: the same key segments, folds and merges.  What differs
// is the way between them.  Here every segment of the layer is at work at once and holds at most two pairs of key tiles, so a
// CTA keeps its K tiles and its Q block in shared memory from the first pass to the second (no second task, no second
// copy), row statistics travel as tagged words that are their own flags (one trip instead of store, fence, count and
// load), the second pass's products wait in tensor memory for the log-sum-exps, which one more K-step then adds, and where
// twice as many CTAs fit the GPU a segment's row halves and tiles go to two of them.
//
// us per call with the sums over heads, general scorer / this one, 32 query heads, 8 KV heads, window 64: 1000 keys 20.5 /
// 16.5, 2304 (the last by halves) 24.0 / 18.2, 3000 25.9 / 20.9, 4608 (the last with one pair a segment) 25.7 / 20.8, 5003
// 31.0 / 26.2, 9216 30.0 / 25.8.  Bound by latency: at 4096 keys the first copy goes out 2 us after the kernel
// before, its products are there 1.5 us later, then 2.7 us of exponentials, 2.5 us until the last CTA's partials are
// merged, 3 us of exponentials, and the way to the next kernel.
//
// A task is (unit, segment[, half]).  CTAs draw tasks from a counter; once none are left, each does the second pass of
// those that it drew, the last one first, whose keys it still holds.  A CTA thus waits for first passes that
// running CTAs have drawn and that wait for nothing: the waits end whatever the number of resident CTAs.  (A cooperative
// launch could do without the counter, but would start only when the kernel before it has left every SM.)
// With halves and an odd number of tiles, the second half of a unit's last segment has no tile in pass 2: that second pass is
// not posted.  So every posted task has products, before which the MMA warp waits for the task's copies.
#pragma once

#include "score_tc.cuh"
#include "tagged.cuh"

namespace skv {

constexpr int kShortTiles = 4;         // key tiles of a segment, at most

struct alignas(64) ShortParams {
  CUtensorMap map_q, map_k;
  float* cols;                         // output of head 0, key 0
  float* row_ent;                      // [unit][kRowBlock] entropy of a row, nats (0: no row)
  unsigned long long* xch;             // tagged words: [unit][segment][kRowBlock] log-sum-exps; kXchPairs later entropies
  int* ctl;
  int* status;
  long long col_stride;
  float c2, inv_c2, v_min;             // |scale| * log2(e), at least 1e-30; 1 / c2; -125 / c2
  int negate, n_keys;
  int window, w_pad, w_shift, group, rows_pg, n_rb;    // as in TcParams
  int n_seg, n_pairs, split, n_tasks;  // segments of a unit, pairs of tiles; 1: a task is one half of a segment of one pair
};

#ifdef __CUDACC__

template <int D>
struct ShortSmem {
  static constexpr int R = kRowBlock;
  static constexpr int kSub = D / 64;                      // 64-column (128-byte) sub-tiles per operand
  static constexpr int kQSub = R * 128, kQBytes = kQSub * kSub;
  static constexpr int kTile = kKeyTile * 128;             // one sub-tile of one key tile
  static constexpr int kKSub = kShortTiles * kTile;        // a sub-tile of all key tiles: any pair is one 256-key operand
  static constexpr int kKOff = kQBytes;
  static constexpr int kOnesOff = kKOff + kKSub * kSub;    // extra K-step, key side: 128 x 16 bf16
  static constexpr int kExtOff = kOnesOff + kKeyTile * 32; // extra K-step, row side: R x 16 bf16
  static constexpr int kPartOff = kExtOff + R * 32;        // [2][3][R] partials (log-sum-exp, entropy)
  static constexpr int kBarOff = kPartOff + 2 * 3 * R * 8;
  enum { kTaskFull = 0, kTaskEmpty = 2, kKFull = 4, kQFull = kKFull + 2, kDone = kQFull + 2, kExtFull, kFold,
         kAccFull = kFold + 4, kAccEmpty = kAccFull + 2, kDrain = kAccEmpty + 2, kCount };
  struct Task { int pass, task, fresh; };                  // pass 0: none left; fresh: its tiles come anew
  struct Work { int unit, g, head, row0, rows, seg, lo, hi, half_lo, half_hi, t_lo, t_hi; };   // head: the unit's first
  struct Flags {
    int abort, mma_in_flight;
    uint32_t tmem;
    unsigned tag;                      // of this launch's words
    unsigned ext_seen;                 // second passes whose log-sum-exps are there
    Task ring[2];
    unsigned short own[kMaxSms];       // tasks whose first pass this CTA has drawn
    Work work[kMaxSms];                // what the tasks are
  };
  static constexpr int kBytes = kBarOff + 8 * kCount + (int)sizeof(Flags);
  static constexpr int kAlloc = kBytes + 1024;             // slack to align the base to 1024 bytes
  static_assert(kAlloc <= 227 * 1024 && kBarOff % 8 == 0, "shared memory of one CTA");
};
constexpr int kShortConsumers = 2 + kComputeWarps;         // MMA, entropies, compute warps

template <int D, int SH>
__global__ void __launch_bounds__(kTcThreads, 1) tc_short(const __grid_constant__ ShortParams p) {
  using L = ShortSmem<D>;
  constexpr int R = L::R;
  static_assert(!Shape<SH>::kNarrow, "wide layouts");
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* sm = smem_raw + (base - raw);
  const uint32_t bars = base + L::kBarOff;
  auto bar = [&](int slot) { return bars + 8u * (uint32_t)slot; };
  auto* const flags = reinterpret_cast<typename L::Flags*>(sm + L::kBarOff + 8 * L::kCount);
  volatile auto* const fl = flags;
  volatile int* const abort_flag = &fl->abort;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int b = 0; b < L::kCount; ++b)
      mbar_init(bar(b), b >= L::kTaskEmpty && b < L::kKFull ? kShortConsumers : b == L::kExtFull ? R / 32
                        : b >= L::kFold && b < L::kAccFull ? 4 : b >= L::kAccEmpty && b < L::kDrain ? kComputeWarps : 1);
    fl->abort = 0;
    fl->mma_in_flight = 0;
    fl->ext_seen = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&p.map_k) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&p.map_q) : "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&flags->tmem)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // operands of pass 2's extra K-step: 1.0 in the first three K columns on the key side, zeros elsewhere
  for (int i = threadIdx.x; i < (kKeyTile + R) * 32 / 16; i += kTcThreads)
    reinterpret_cast<uint4*>(sm + L::kOnesOff)[i] =
        i < kKeyTile * 2 && (i & 8) == 0 ? make_uint4(0x3f803f80u, 0x00003f80u, 0u, 0u) : make_uint4(0u, 0u, 0u, 0u);
  // What the tasks are: divisions, and parameters that no cache holds yet, while the kernel before still runs.  (Each role
  // working them out after the wait, and every warp reading the launch's tag: a CTA's first copy went out 5000 to 6200 clocks
  // after the wait, now 3600 to 4100.)
  const int n_keys = p.n_keys, n_tiles = (n_keys + kKeyTile - 1) / kKeyTile, per_unit = p.n_seg << p.split;
  for (int task = threadIdx.x; task < p.n_tasks; task += kTcThreads) {
    typename L::Work w;
    w.unit = task / per_unit;
    const int at = task - w.unit * per_unit;
    w.seg = at >> p.split;
    w.g = w.unit / p.n_rb;
    w.row0 = (w.unit - w.g * p.n_rb) * R;
    w.rows = min(R, p.rows_pg - w.row0);
    w.head = w.g * p.group + w.row0 / p.w_pad;
    w.lo = 2 * (int)((unsigned)w.seg * (unsigned)p.n_pairs / (unsigned)p.n_seg);       // tiles [lo, hi), whole pairs
    w.hi = 2 * (int)((unsigned)(w.seg + 1) * (unsigned)p.n_pairs / (unsigned)p.n_seg);
    w.half_lo = at & p.split;                              // row halves of pass 1
    w.half_hi = p.split ? w.half_lo + 1 : w.rows > 128 ? 2 : 1;
    w.t_lo = w.lo + w.half_lo;                             // tiles of pass 2, possibly none
    w.t_hi = min(n_tiles, p.split ? w.t_lo + 1 : w.hi);
    flags->work[task] = w;
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = flags->tmem;
  pdl_trigger();
  pdl_wait();          // inputs, counters and exchange words belong to the kernels before this one until here

  auto words_of = [&](int unit, int seg) { return p.xch + (size_t)(unit * p.n_seg + seg) * R; };
  constexpr size_t kEntWords = kXchPairs;
  auto is_row = [&](int row) { return row < p.rows_pg && (row & (p.w_pad - 1)) < p.window; };   // row of the KV group, padding excluded
  auto next_task = [&](int n, typename L::Task& t) {
    int ok = 1;
    if (lane == 0)
      ok = mbar_wait(bar(L::kTaskFull + (n & 1)), (uint32_t)(n >> 1) & 1u, abort_flag) ? 1 : 0;
    if (!__shfl_sync(0xffffffffu, ok, 0)) return false;
    asm volatile("" ::: "memory");
    t = flags->ring[n & 1];
    asm volatile("" ::: "memory");
    __syncwarp();
    if (lane == 0) mbar_arrive(bar(L::kTaskEmpty + (n & 1)));
    return t.pass != 0;
  };
  // Bounds a poll of exchange words: false once the CTA gives up.
  auto keep_polling = [&](long long& t0) {
    if (*abort_flag) return false;
    const long long now = clock64();
    if (t0 == 0) t0 = now;
    if ((unsigned long long)(now - t0) > kWaitCycles) { *abort_flag = 1; return false; }
    return true;
  };
  // Words s0, s0 + 1, ... of a row (a segment each) once all of them are there.
  auto read_words = [&](const unsigned long long* words, unsigned tag, int s0, auto& v, long long& t0) {
    constexpr int N = sizeof(v) / sizeof(float);
    for (;;) {
      bool all = true;
#pragma unroll
      for (int b = 0; b < N; ++b) {
        const unsigned long long x = s0 + b < p.n_seg ? get_word(words + (size_t)(s0 + b) * R) : (unsigned long long)tag << 32;
        all = all && word_has(x, tag);
        v[b] = word_value(x);
      }
      if (all) return true;
      if (!keep_polling(t0)) return false;
    }
  };
  // Merges partials s0, s0 + 1, ... of a row into (M, W, X).
  auto merge_words = [&](float& M, float& W, float& X, const float* l, const float* h, int s0) {
    float2 pv[kMergeGroup];
#pragma unroll
    for (int b = 0; b < kMergeGroup; ++b) pv[b] = s0 + b < p.n_seg ? make_float2(l[b], h ? h[b] : 0.f) : make_float2(-INFINITY, 0.f);
    merge_partials(M, W, X, pv);
  };

  if (warp == 0) {
    // ---------------- tasks and copies ----------------
    if (lane == 0) {
      const uint64_t pol = l2_policy_evict_normal();
      int* const ticket = p.ctl + kCtlTicket;
      int n_own = 0, loaded = -1;
      unsigned loads = 0;
      const unsigned before = (unsigned)__ldcg(p.ctl + kCtlTag);   // one thread reads it: by all warps of all CTAs it took 2000 clocks
      int tk = atomicAdd(ticket, 1);
      flags->tag = before + 1u;
      for (int n = 0;; ++n) {
        typename L::Task t{0, 0, 0};
        if (tk < p.n_tasks) {
          t.pass = 1;
          t.task = tk;
          flags->own[n_own++] = (unsigned short)tk;
        } else {
          while (t.pass == 0 && n_own > 0) {
            t.task = flags->own[--n_own];
            if (flags->work[t.task].t_lo < flags->work[t.task].t_hi) t.pass = 2;
          }
        }
        t.fresh = t.pass != 0 && t.task != loaded;
        if (!mbar_wait(bar(L::kTaskEmpty + (n & 1)), ((uint32_t)(n >> 1) & 1u) ^ 1u, abort_flag)) break;
        flags->ring[n & 1] = t;
        mbar_arrive(bar(L::kTaskFull + (n & 1)));
        if (t.pass == 0) break;
        if (t.fresh) {
          // The copies before have landed, and the MMAs of the task before have read what they wanted.  (No wait here or in
          // the MMA warp can be two phases behind, whose parity would let it through: a task's first products wait for its
          // copies' first pair of tiles, and those copies for the products of the task before and for all copies before.)
          bool ok = n == 0 || mbar_wait(bar(L::kDone), (uint32_t)(n - 1) & 1u, abort_flag);
          for (int b = L::kKFull; b < L::kDone && ok && loads > 0; ++b)
            ok = mbar_wait(bar(b), (loads - 1u) & 1u, abort_flag);
          if (!ok) break;
          const typename L::Work w = flags->work[t.task];
          auto load_q = [&](int hq) {
            mbar_expect_tx(bar(L::kQFull + hq), L::kQBytes / 2);
            for (int c = 0; c < L::kSub; ++c)
              tma_load_3d_hint(base + c * L::kQSub + hq * (128 * 128), &p.map_q, bar(L::kQFull + hq), c * 64, hq * 128 & (p.w_pad - 1),
                               w.head + (hq * 128 >> p.w_shift), pol);
          };
          // a tile may reach beyond the last key (into zero fill): the causal mask discards those keys
          auto load_k = [&](int pair) {
            mbar_expect_tx(bar(L::kKFull + pair), 2 * L::kTile * L::kSub);
            for (int i = 2 * pair; i < 2 * pair + 2; ++i)
              for (int c = 0; c < L::kSub; ++c)
                tma_load_3d_hint(base + L::kKOff + c * L::kKSub + i * L::kTile, &p.map_k, bar(L::kKFull + pair), c * 64,
                                 (w.lo + i) * kKeyTile, w.g, pol);
          };
          load_k(0);
          load_q(w.half_lo);
          load_q(1 - w.half_lo);
          if (w.hi - w.lo > 2) load_k(1);
          else mbar_arrive(bar(L::kKFull + 1));
          loaded = t.task;
          ++loads;
        }
        if (t.pass == 1) {
          // the next task once this one's products are done: CTAs that start later come first
          if (!mbar_wait(bar(L::kDone), (uint32_t)n & 1u, abort_flag)) break;
          tk = atomicAdd(ticket, 1);
        }
      }
      // every copy this thread issued must have landed before the CTA may exit
      if (loads)
        for (int b = L::kKFull; b < L::kDone; ++b) mbar_drain(bar(b), (loads - 1u) & 1u, abort_flag);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    if (lane == 0) {
      constexpr uint32_t idesc_ext = instr_desc(128, R);
      const uint32_t idesc = idesc_ext | (p.negate ? 1u << 13 : 0u);
      const uint64_t q_desc0 = smem_desc(base), k_desc0 = smem_desc(base + L::kKOff);
      const uint64_t ones_desc = smem_desc_k16(base + L::kOnesOff), ext_desc = smem_desc_k16(base + L::kExtOff);
      unsigned loads = 0, u = 0, n_ext = 0;                // copies, accumulators, second passes so far
      bool ok = true;
      auto wait = [&](int b, unsigned parity) { return mbar_wait(bar(b), parity & 1u, abort_flag); };
      auto acc_free = [&]() {
        const bool r = wait(L::kAccEmpty + (u & 1), (u >> 1) ^ 1u);
        tc_fence_after();
        return r;
      };
      for (int n = 0; ok; ++n) {
        if (!wait(L::kTaskFull + (n & 1), (unsigned)n >> 1)) break;
        asm volatile("" ::: "memory");
        const typename L::Task t = flags->ring[n & 1];
        asm volatile("" ::: "memory");
        mbar_arrive(bar(L::kTaskEmpty + (n & 1)));
        if (t.pass == 0) break;
        const typename L::Work w = flags->work[t.task];
        loads += t.fresh;
        if (t.pass == 1) {
          // accumulator = (pair, row half): A = one 128-row half of Q, B = the pair's 256 keys
          for (int pr = 0; 2 * pr < w.hi - w.lo && ok; ++pr)
            for (int hf = w.half_lo; hf < w.half_hi; ++hf, ++u) {
              if (!(ok = wait(L::kKFull + pr, loads - 1u) && wait(L::kQFull + hf, loads - 1u) && acc_free())) break;
#pragma unroll
              for (int kk = 0; kk < D / 16; ++kk) {
                const uint32_t qo = (kk / 4) * L::kQSub + hf * (128 * 128) + (kk % 4) * 32;
                const uint32_t ko = (kk / 4) * L::kKSub + 2 * pr * L::kTile + (kk % 4) * 32;
                tc_mma_bf16(tmem + (u & 1) * 256, q_desc0 + (qo >> 4), k_desc0 + (ko >> 4), idesc, kk > 0);
              }
              fl->mma_in_flight = 1;
              tc_commit(bar(L::kAccFull + (u & 1)));
            }
        } else {
          // accumulator = one key tile: A = 128 keys, B = the whole Q block.  Two tiles' products are on their way before the
          // log-sum-exps are there; one more K-step then adds -lse / c2 of every row: ones (key side) x three
          // bf16 pieces of the value (row side).
          const int tiles = w.t_hi - w.t_lo;
          auto products = [&](int i) {
            if (!(ok = wait(L::kKFull + (w.t_lo + i - w.lo) / 2, loads - 1u) && wait(L::kQFull, loads - 1u) &&
                       wait(L::kQFull + 1, loads - 1u) && acc_free())) return;
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) {
              const uint32_t ko = (kk / 4) * L::kKSub + (w.t_lo + i - w.lo) * L::kTile + (kk % 4) * 32;
              const uint32_t qo = (kk / 4) * L::kQSub + (kk % 4) * 32;
              tc_mma_bf16(tmem + (u & 1) * 256, k_desc0 + (ko >> 4), q_desc0 + (qo >> 4), idesc, kk > 0);
            }
            fl->mma_in_flight = 1;
            ++u;
          };
          products(0);
          for (int i = 0; i < tiles && ok; ++i) {
            if (i == 0) {
              if (tiles > 1) products(1);
              if (!ok || !(ok = mbar_wait(bar(L::kExtFull), n_ext & 1u, abort_flag))) break;
              fl->ext_seen = n_ext + 1;
            } else if (i > 1) {
              products(i);
              if (!ok) break;
            }
            const unsigned at = i == 0 && tiles > 1 ? u : u + 1;    // of accumulator u - 1, or, of the first of two, u - 2
            tc_mma_bf16(tmem + (at & 1) * 256, ones_desc, ext_desc, idesc_ext, 1);
            tc_commit(bar(L::kAccFull + (at & 1)));
          }
          ++n_ext;
        }
        if (!ok) break;
        tc_commit(bar(L::kDone));
      }
      // all issued MMAs must retire before tensor memory is freed
      if (fl->mma_in_flight) {
        tc_commit(bar(L::kDrain));
        if (mbar_drain(bar(L::kDrain), 0, abort_flag)) fl->mma_in_flight = 0;
      }
    }
  } else if (warp == 2) {
    // ---------------- entropies, beside the second pass: a unit's rows are dealt out to its segments' CTAs ----------------
    typename L::Task t;
    unsigned n_ext = 0;
    for (int n = 0; next_task(n, t); ++n) {
      const typename L::Work w = flags->work[t.task];
      if (t.pass != 2) continue;
      ++n_ext;
      if (p.split && w.half_lo != 0) continue;
      const unsigned tag = flags->tag;
      long long t0 = 0;
      for (int r = w.seg * R / p.n_seg + lane; r < (w.seg + 1) * R / p.n_seg; r += 32) {
        float ent = 0.f;
        if (is_row(w.row0 + r)) {
          const unsigned long long* const words = words_of(w.unit, 0) + r;
          float M = -INFINITY, W = 0.f, X = 0.f;
          for (int s0 = 0; s0 < p.n_seg; s0 += kMergeGroup) {
            float l[kMergeGroup], h[kMergeGroup];
            if (!read_words(words + kEntWords, tag, s0, h, t0) || !read_words(words, tag, s0, l, t0)) break;
            merge_words(M, W, X, l, h, s0);
          }
          if (W > 0.f) ent = kLn2 * (__log2f(W) + X / W);
        }
        p.row_ent[(size_t)w.unit * R + r] = ent;
      }
    }
    // No task is left and, once the last log-sum-exps are there, no word is read any more: the CTA signs off beside its last
    // exponentials (by all of its warps after them: 0.4 us later).  The last one leaves the counters as it found them, and
    // the tags one further.
    int last = 0;
    if (lane == 0) {
      long long t0 = 0;
      while (fl->ext_seen != n_ext && keep_polling(t0)) {}
      last = atomicAdd(p.ctl + kCtlExit, 1) == (int)gridDim.x - 1;
      if (last) p.ctl[kCtlTicket] = 0;
    }
    if (__shfl_sync(0xffffffffu, last, 0)) pass_tags_on(p.xch, p.ctl, flags->tag, lane, 32);
  } else if (warp >= kHelperWarps) {
    // ---------------- compute warps ----------------
    const int quarter = warp & 3;            // tensor-memory lane quarter this warp may read
    const int sub = (warp - kHelperWarps) >> 2;   // which quarter of an accumulator's columns it takes
    const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
    float2* const part_s = reinterpret_cast<float2*>(sm + L::kPartOff);
    const int ct = (int)threadIdx.x - kHelperWarps * 32, row_lo = quarter * 32 + lane;
    const uint64_t c22 = pack2(p.c2, p.c2);
    const int last_open_key = n_keys - p.window;           // the last key every window row sees
    unsigned u = 0, n_fold = 0;
    auto acc_full = [&]() {
      const uint32_t b = bar(L::kAccFull + (u & 1)), parity = (u >> 1) & 1u;
      bool ok = mbar_try(b, parity);
      if (!__all_sync(0xffffffffu, ok)) ok = __all_sync(0xffffffffu, mbar_wait(b, parity, abort_flag)) != 0;
      tc_fence_after();
      return ok;
    };
    auto acc_release = [&]() {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(L::kAccEmpty + (u & 1)));
    };
    auto acc_addr = [&]() { return lane_base + (u & 1) * 256; };
    // -lse / c2 of a row as hi + mid + lo (bf16 each: 24 bits together) into the extra K-step's operand; rows
    // that do not exist get a huge negative value so that their 2^x is 0.
    auto put_lse = [&](int r, float nlse) {
      const float Lv = nlse == -INFINITY ? kMaskedAcc : nlse * p.inv_c2;
      const __nv_bfloat16 hi = __float2bfloat16_rn(Lv);
      const float r1 = Lv - __bfloat162float(hi);
      const __nv_bfloat16 mid = __float2bfloat16_rn(r1);
      const __nv_bfloat16 lo = __float2bfloat16_rn(r1 - __bfloat162float(mid));
      unsigned char* bx = sm + L::kExtOff;
      *reinterpret_cast<__nv_bfloat16*>(bx + k16_offset(r, 0)) = hi;
      *reinterpret_cast<__nv_bfloat16*>(bx + k16_offset(r, 1)) = mid;
      *reinterpret_cast<__nv_bfloat16*>(bx + k16_offset(r, 2)) = lo;
    };
    bool live = true;
    typename L::Task t;
    for (int n = 0; live && next_task(n, t); ++n) {
      const typename L::Work w = flags->work[t.task];
      const unsigned tag = flags->tag;
      if (t.pass == 1) {
        // This thread owns row (quarter * 32 + lane) of the halves and the keys [sub * 64, sub * 64 + 64) of every pair.
        const int n_half = w.half_hi - w.half_lo, n_acc = (w.hi - w.lo) / 2 * n_half;
        if (n_half <= 0) continue;
        float v[32] = {};
        auto chunk = [&](RowStat& r, int jb, bool first, int hf) {
          bool careful = jb + 31 > last_open_key;          // holds window keys, or lies beyond the sequence
          if (first && !careful) {                         // a segment's first chunk gives the rows their reference
            float mx = v[0];
#pragma unroll
            for (int e = 1; e < 32; ++e) mx = fmaxf(mx, v[e]);
            r.ref = mx * p.c2;
          }
          const RowStat before = r;
          if (!careful) careful = __any_sync(0xffffffffu, !stat_add(r, v, c22));
          if (careful) {
            r = before;
            stat_add_masked(r, v, p.c2, jb, last_open_key + ((hf * 128 + row_lo) & (p.w_pad - 1)));
          }
        };
        RowStat rs[2] = {{-INFINITY, 0.f, 0.f}, {-INFINITY, 0.f, 0.f}};
        for (int k = 0; k < n_acc; ++k) {
          if (!acc_full()) { live = false; break; }
          const int it = n_half == 2 ? k >> 1 : k, hf = n_half == 2 ? k & 1 : w.half_lo;
          const int jb = (w.lo + 2 * it) * kKeyTile + sub * 64;
          const bool warp_active = hf * 128 + quarter * 32 < w.rows;
          // (one copy of the body: with two, 2304 keys with all statistics take 17.8 us instead of 16.9, 4096 20.4 instead of 19.9)
#pragma unroll 1
          for (int c = 0; c < 2; ++c) {
            if (warp_active) tmem_ld(acc_addr() + sub * 64 + 32 * c, v);
            if (c == 1) acc_release();
            if (warp_active) chunk(rs[0], jb + 32 * c, it == 0 && c == 0, hf);
          }
          if (n_half == 2) {
            const RowStat o = rs[0];
            rs[0] = rs[1];
            rs[1] = o;
          }
          ++u;
        }
        if (!live) break;
        // the four warps of a lane quarter meet; column group 0 folds the rows of the first (or only) half, column group 1
        // those of the second
        float2* const buf = part_s + (n_fold & 1) * 3 * R;
        const float2 part0 = stat_partial(rs[0]), part1 = stat_partial(rs[1]);
        if (sub != 0) buf[(sub - 1) * R + row_lo] = part0;
        if (n_half == 2 && sub != 1) buf[(sub == 0 ? 0 : sub - 1) * R + 128 + row_lo] = part1;
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(L::kFold + quarter));
        if (!__all_sync(0xffffffffu, mbar_wait(bar(L::kFold + quarter), n_fold & 1u, abort_flag))) break;
        ++n_fold;
        if (sub < n_half) {
          const float2 f = fold_row(buf + sub * 128 + row_lo, R, sub == 0 ? part0 : part1, sub);
          unsigned long long* const to = words_of(w.unit, w.seg) + (w.half_lo + sub) * 128 + row_lo;
          put_word(to, tagged(f.x, tag));
          put_word(to + kEntWords, tagged(f.y, tag));
        }
        continue;
      }
      // Pass 2: the unit's log-sum-exps, a thread per row, all partials of a row in one round of loads, merged in the
      // groups of score_tc.cuh.  At first one word alone is polled: with all threads reading all of their words over and over
      // the words themselves were late.
      if (ct < R) {
        bool ok = true;
        float nlse = -INFINITY;
        if (is_row(w.row0 + ct)) {
          const unsigned long long* const words = words_of(w.unit, 0) + ct;
          float M = -INFINITY, W = 0.f, X = 0.f, first[1];
          long long t0 = 0;
          constexpr int kRounds = 3;
          ok = read_words(words, tag, p.n_seg - 1, first, t0);
          for (int s0 = 0; s0 < p.n_seg && ok; s0 += kRounds * kMergeGroup) {
            float l[kRounds * kMergeGroup];
            ok = read_words(words, tag, s0, l, t0);
#pragma unroll
            for (int k = 0; k < kRounds; ++k) merge_words(M, W, X, l + k * kMergeGroup, nullptr, s0 + k * kMergeGroup);
          }
          if (W > 0.f) nlse = -(M + __log2f(W));
        }
        if (!__all_sync(0xffffffffu, ok)) break;
        put_lse(ct, nlse);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // visible to the tensor core
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(L::kExtFull));
      }
      // This thread owns key (tile * 128 + quarter * 32 + lane); x = c2 * accumulator.  Columns (rows of the block) this
      // warp sums: a quarter of them on every tile, or, where a head spans more, the head's rows on every second or
      // fourth tile, so that a head's column sum never spans two warps.
      const float v_min = p.v_min, inv_w = 1.0f / (float)p.window;
      constexpr int kW = Shape<SH>::kW, kCols = kW <= 64 ? 64 : kW;
      const int turn = kW == 256 ? 3 : kW == 128 ? 1 : 0;
      const int col0 = kW == 256 ? 0 : kW == 128 ? (sub & 1) * 128 : sub * 64;
      const int my_turn = kW == 128 ? sub >> 1 : sub;
      const bool warp_active = col0 < w.rows;
      const int h0 = (w.row0 + col0) >> p.w_shift;         // heads within the KV group
      float* const cols = p.cols + (size_t)w.g * p.group * p.col_stride;
      for (int tile = w.t_lo; tile < w.t_hi; ++tile) {
        if (!acc_full()) { live = false; break; }
        const int j = tile * kKeyTile + quarter * 32 + lane;
        const bool plain = (tile + 1) * kKeyTile - 1 <= last_open_key;   // all of its keys are visible to every window row
        const int i_min = j - last_open_key;               // window rows i < i_min do not see key j
        const bool mine = warp_active && ((int)u & turn) == (my_turn & turn);
        const uint32_t taddr = acc_addr() + col0;
        float tot = 0.f;
        int head = h0;
#pragma unroll 2
        for (int c = 0; c < kCols; c += 32) {
          float v[32] = {};
          if (mine) tmem_ld(taddr + c, v);
          if (c == kCols - 32) acc_release();              // every load of the tile has landed
          if (!mine) continue;
          if (!plain) {
#pragma unroll
            for (int e = 0; e < 32; ++e)
              if (((col0 + c + e) & (p.w_pad - 1)) < i_min) v[e] = kMaskedAcc;
          }
          auto finish_head = [&]() {
            if (head < p.group && j < n_keys) cols[(size_t)head * p.col_stride + j] = tot * inv_w;
            ++head;
            tot = 0.f;
          };
          if constexpr (kW == 16) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              tot += sum_exp<8>(v + 8 * k, c22, v_min, 4 * k);
              if (((c + 8 * k + 8) & (p.w_pad - 1)) == 0) finish_head();
            }
          } else {
            tot += sum_exp<32>(v, c22, v_min);
            if (((c + 32) & (kW - 1)) == 0) finish_head();
          }
        }
        ++u;
      }
    }
  }

  // ---------------- teardown ----------------
  tc_fence_before();
  __syncthreads();
  if (*abort_flag && threadIdx.x == 0) atomicCAS(p.status, 0, (int)STRUCTKV_ERR_TIMEOUT);
  // tensor memory is freed only when no MMA of this CTA can still write to it
  if (warp == 1 && !fl->mma_in_flight) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

template <int D, int SH>
cudaError_t short_launch(const ShortParams& p, int grid, int device, cudaStream_t st) {
  auto kern = tc_short<D, SH>;
  constexpr int kAlloc = ShortSmem<D>::kAlloc;
  static std::atomic<unsigned long long> ready{0};        // devices whose shared-memory limit has been raised
  const unsigned long long bit = 1ull << (device & 63);
  if (!(ready.load(std::memory_order_acquire) & bit)) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kAlloc);
    if (e != cudaSuccess) return e;
    ready.fetch_or(bit, std::memory_order_release);
  }
  return launch_pdl(kern, dim3(grid), dim3(kTcThreads), kAlloc, st, p);
}
template <int D>
cudaError_t short_dispatch(int shape, const ShortParams& p, int grid, int device, cudaStream_t st) {
  switch (shape) {
    case kWide16: return short_launch<D, kWide16>(p, grid, device, st);
    case kWide32: return short_launch<D, kWide32>(p, grid, device, st);
    case kWide64: return short_launch<D, kWide64>(p, grid, device, st);
    case kWide128: return short_launch<D, kWide128>(p, grid, device, st);
    case kWide256: return short_launch<D, kWide256>(p, grid, device, st);
  }
  return cudaErrorInvalidValue;
}
#endif  // __CUDACC__

// One translation unit per head dimension instantiates the kernels.
cudaError_t short_launch_64(int shape, const ShortParams& p, int grid, int device, cudaStream_t st);
cudaError_t short_launch_128(int shape, const ShortParams& p, int grid, int device, cudaStream_t st);

}  // namespace skv
