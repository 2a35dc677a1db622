// Tensor-core scorer of short windows (up to 32 score rows per KV group): K is read ONCE.
//
// A column sum needs the normaliser of every row, so the general scorer (score_tc.cuh) computes all logits twice
// and reads K twice; with few rows per key that reading is what bounds it.  Here a team of G CTAs shares a unit (the score
// rows of one KV group) by keys, and a CTA holds the unit's logits over its own keys in tensor memory, 32 columns for
// 128 keys, from the first pass over them until the team knows the rows' normalisers: at 32768 keys 7 of 16
// tiles a unit, two units in flight and the keys of the next ones on their way.
// us per layer with the sums over heads, general scorer / this one, 32 query heads, 8 KV heads, window 8, 32 layers: 2500 keys
// 3.2 / 3.5, 5003 4.1 / 3.9, 9001 6.8 / 4.3, 20011 13.8 / 8.4, 32768 21 / 12.6 (reading K once takes 10.4), 98304 67 / 39,
// 131072 93 / 53, 262144 183 / 121; one layer of 32768 37.4 / 30.9, of 98304 76.7 / 60.4.  What is left above the reading is the way from tile to tile of a warp, at 60 % of the
// special-function unit's rate.  With 64 rows (window 16) both forms take as long: there the exponentials bound it.
//
// How a team adds up its rows' statistics, without fences, flags or a second trip:
//   direct (teams of up to kDirectTeam)  every CTA leaves its partials as words that carry a tag, reads
//           all of its mates' and merges them in order
//   summed (larger teams)                a row has one reference for the whole team (its largest logit over a few
//           sampled keys; one CTA finds a unit's, some units ahead, and leaves them as tagged words), so that sums of
//           2^(x - ref) add up; they do as fixed-point integers, in any order the same bits, in words whose
//           top byte counts the CTAs.  Where a CTA's sum leaves the range
//           (a logit 2^20 above the reference) it marks the word, and the team takes the direct way for that unit.
// The more mates, the more words a direct team reads.  us per layer, direct / summed, one layer | one of 32: 74 CTAs (65536
// keys) - | 31.6 / 26.7; 37 CTAs (8 KV heads, 20011 keys) 28.8 / 26.7 | 9.8 / 8.4, (32768 keys) 33.1 / 30.8 | 13.9 /
// 12.7, (4 KV heads, 4096 keys) 20.6 / 18.5 | 3.8 / 2.7; 24 CTAs (6 KV heads, 5003 keys) 21.0 / 19.9 | 4.0 / 3.1.  The
// general scorer takes 18.5 | 2.9 for those 4096 keys and 20.4 | 4.3 for those 5003, so direct teams of 24 and more lost.
// Those of 18 do not (8 KV heads, 4096 keys 20.3 | 3.4, general 21.3 | 4.5) and keep their form: summed they take 18.8 | 3.0,
// but their columns' errors against float64 are 3 to 8 % larger (3.9e-7 instead of 3.7e-7; of teams of 37 4.2e-7
// instead of 4.5e-7).  The references came from a launch of
// their own at first, which a layer by itself waited for; us with it / with them found inside, one layer: 8 KV heads
// 40000 keys 43.0 / 36.6, 98304 64.6 / 60.1, 262144 150 / 135; 4 KV heads 40000 32.9 / 26.7, 131072 49.5 / 44.4;
// one KV head 32768 24.4 / 18.5; a layer of 32 with 8 KV heads of 262144 keys 135 / 121.
// Which keys a CTA holds depends on the sequence length, the KV heads and the SM count alone: results depend
// neither on timing nor on how many layers a call has.
//
// All CTAs of the launch must run at once (the members of a team wait for one another): the launch is
// cooperative.  Every wait is bounded, as in score_tc.cuh.
//
// Warps: 0-15 compute (lane quarter = warp & 3; each does a unit's column sums as soon as its normalisers are there, else
// the statistics of its next unit as soon as the MMAs have left it), 16 = TMA producer, 17 = MMA issuer, 18 = waits
// for the team's normalisers, 19 = folds and publishes this CTA's statistics.
#pragma once

#include "score_tc.cuh"
#include "tagged.cuh"

namespace skv {

constexpr int kResSubs = 4;            // compute warps of a lane quarter
constexpr int kResWarps = 4 * kResSubs;
constexpr int kResThreads = (kResWarps + 4) * 32;   // 20 warps: the most that fit at 96 registers a thread
constexpr int kResChunk = 32;          // keys are dealt out to a team's CTAs in chunks of 32
constexpr int kResRing = 8;            // units a CTA may have between its statistics and its last column sum
constexpr int kRefAhead = 2 * kResRing;   // a unit's common references are found so many units before
// A row's summed words: [63:56] CTAs so far, [55] somebody's sum is out of range, below it sum Z in units of
// 2^-26; [63:56] CTAs, below it sum (U + 2^21) in units of 2^-26.
constexpr float kSumUnit = 67108864.f, kSumLimit = 2097152.f;
constexpr unsigned long long kSumCount = 1ull << 56, kSumOver = 1ull << 55, kSumBias = 1ull << 47;
static_assert(kMaxSms * 2097152ull * 67108864ull < kSumOver && kMaxSms * 2 * kSumBias < kSumCount, "summed words");
static_assert(kXchSlots > 2 * kResRing, "slots of tagged words");
static_assert(kRefSlots >= kRefAhead + 2 * kResRing && kRefAhead <= kDirectTeam, "rings of references");

struct ResProblem {
  float* cols;                         // output of head 0, key 0
  const __nv_bfloat16 *q, *k;
  int n_keys;
  float c2;                            // |scale| * log2(e), at least 1e-30
  int negate;
};
// The same with this CTA's share of the keys: chunks [lo, lo + c), tiles of up to four.
struct ResShare { ResProblem p; int lo, c; };
template <int MAXP>
struct alignas(64) ResParams {
  CUtensorMap map_q[MAXP], map_k[MAXP];
  ResProblem prob[MAXP];
  int n_prob, n_kv, team, teams;       // CTAs of a team, teams
  int window, w_pad, group, rows_pg;   // rows_pg = group * w_pad <= kResRows
  int* ctl;
  unsigned long long* xch;             // tagged words, kXchWords
  unsigned long long* sums;            // summed: [unit of the launch][kResRows] x {Z, U}; NULL: direct
  float* row_ent;                      // [problem][KV group][kRowBlock] entropy of a row, nats (0: no row)
  long long col_stride, k_stride_head, k_stride_token;   // elements
  int* status;
};

#ifdef __CUDACC__

template <int D, int MAXP>
struct ResSmem {
  static constexpr int kSub = D / 64;                      // 64-column (128-byte) sub-tiles per operand
  static constexpr int R = kResRows;
  static constexpr int kStages = 6;                        // K tiles on their way
  static constexpr int kSlots = 512 / R;                   // tiles in tensor memory
  static constexpr int kTileSub = 128 * 128;               // one sub-tile of a K tile: 128 keys x 128 bytes
  static constexpr int kTile = kTileSub * kSub;
  static constexpr int kQSub = R * 128;
  static constexpr int kQ = kQSub * kSub;
  static constexpr int kQOff = kStages * kTile;
  static constexpr int kStatOff = kQOff + 2 * kQ;          // [ring][quarter][R] {ref, Z, U} of a lane quarter's keys
  static constexpr int kLseOff = kStatOff + kResRing * 4 * R * 12;   // [ring][R] -log2-sum-exp of a row (-inf: no row)
  static constexpr int kProbOff = kLseOff + kResRing * R * 4;
  static constexpr int kBarOff = kProbOff + MAXP * (int)sizeof(ResShare);
  enum { kKFull = 0, kKEmpty = kStages, kQFull = 2 * kStages, kQEmpty = kQFull + 2, kFull = kQEmpty + 2, kFree = kFull + kSlots,
         kStats = kFree + kSlots, kDrain = kStats + kResRing, kCount };
  // What the compute warps and those that wait for the team tell one another.
  struct Flags {
    int abort, mma_in_flight, last;
    uint32_t tmem;
    int summed;                        // units whose column sums are done
    int known;                         // units whose normalisers are there
    int sum_ctr[kResRing];             // warps that are done with a unit's sums
  };
  static constexpr int kBytes = kBarOff + 8 * kCount + (int)sizeof(Flags);
  static constexpr int kAlloc = kBytes + 1024;             // slack to align the base to 1024 bytes
  static_assert(kAlloc <= 227 * 1024 && kProbOff % 8 == 0 && kBarOff % 8 == 0, "shared memory of one CTA");
};

template <int D, int MAXP>
__global__ void __launch_bounds__(kResThreads, 1) tc_resident(const __grid_constant__ ResParams<MAXP> p) {
  using L = ResSmem<D, MAXP>;
  constexpr int R = kResRows, kStages = L::kStages, kSlots = L::kSlots;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* sm = smem_raw + (base - raw);
  const uint32_t bars = base + L::kBarOff;
  auto bar = [&](int slot) { return bars + 8u * (uint32_t)slot; };
  auto* const flags = reinterpret_cast<typename L::Flags*>(sm + L::kBarOff + 8 * L::kCount);
  volatile auto* const fl = flags;
  volatile int* const abort_flag = &fl->abort;
  float* const stat_s = reinterpret_cast<float*>(sm + L::kStatOff);
  float* const lse_s = reinterpret_cast<float*>(sm + L::kLseOff);
  ResShare* const prob_s = reinterpret_cast<ResShare*>(sm + L::kProbOff);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int G = p.team, team = blockIdx.x / G, rank = blockIdx.x - team * G;

  if (threadIdx.x == 0) {
    for (int b = 0; b < L::kCount; ++b) mbar_init(bar(b), b >= L::kStats && b < L::kDrain ? kResWarps : b >= L::kFree && b < L::kStats ? 4 : 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = threadIdx.x; i < (int)(sizeof(typename L::Flags) / 4); i += kResThreads) reinterpret_cast<int*>(flags)[i] = 0;
  for (int i = threadIdx.x; i < p.n_prob; i += kResThreads) {
    const int chunks = (p.prob[i].n_keys + kResChunk - 1) / kResChunk, lo = rank * chunks / G;
    prob_s[i] = ResShare{p.prob[i], lo, (rank + 1) * chunks / G - lo};
  }
  __syncthreads();
  if (warp == kResWarps + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&flags->tmem)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = flags->tmem;
  pdl_trigger();
  pdl_wait();          // inputs, exchange words and output buffers belong to the kernels before this one until here

  const int n_kv = p.n_kv, n_prob = p.n_prob, teams = p.teams;
  const unsigned tag0 = (unsigned)__ldcg(p.ctl + kCtlTag) + 1u;      // unit u of this team carries tag0 + u
  // Every role walks the team's KV groups gu = team, team + teams, ... of all problems: unit 0, 1, ...
  struct Walk { int pi, g; };                              // KV group g of problem pi
  auto walk_from = [&]() { return Walk{team / n_kv, team % n_kv}; };
  auto walk_on = [&](Walk& w) {
    for (w.g += teams; w.g >= n_kv; w.g -= n_kv) ++w.pi;
  };
  auto unit_of = [&](const Walk& w) { return w.pi * n_kv + w.g; };   // of the launch
  auto is_row = [&](int row) { return row < p.rows_pg && (row & (p.w_pad - 1)) < p.window; };
  auto stat_at = [&](unsigned u, int quarter, int row) { return stat_s + ((u % kResRing * 4 + quarter) * R + row) * 3; };
  // Bounds a poll: false once the CTA gives up.
  auto keep_polling = [&](long long& t0) {
    if (*abort_flag) return false;
    const long long now = clock64();
    if (t0 == 0) t0 = now;
    if ((unsigned long long)(now - t0) > kWaitCycles) { *abort_flag = 1; return false; }
    return true;
  };
  // Tagged words of unit u: [team][slot][rank][row], log-sum-exps, then entropies.  Who publishes unit v has summed, so
  // known, unit v - kResRing; so every CTA had published that one, hence summed and known unit v - 2 kResRing.  Knowing
  // a unit means that its log-sum-exps have been read.  The CTA that leaves its entropies reads those afterwards, before it
  // looks at the next unit: all words are read of units before v - 2 kResRing, so that a slot must
  // last one unit longer than two rings.
  constexpr size_t kEntWords = kXchPairs;
  // (Who walks the units counts the slots along: 17 is no power of two.)
  auto tagged_words = [&](int slot, int row) { return p.xch + ((size_t)(team * kXchSlots + slot) * G * R + row); };
  auto next_slot = [](int slot) { return slot + 1 < kXchSlots ? slot + 1 : 0; };
  // This CTA's statistics of a row, its lane quarters' in order, relative to `ref`.
  auto fold = [&](unsigned u, int row, float ref) {
    RowStat f{ref, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float* st = stat_at(u, k, row);
      const float e = st[0] - ref, m = st[0] == ref ? 1.f : st[0] == -INFINITY ? 0.f : fast_exp2(e);
      f.Z = fmaf(m, st[1], f.Z);
      if (st[0] != -INFINITY) f.U += m * fmaf(e, st[1], st[2]);
    }
    return f;
  };
  auto publish = [&](unsigned u, int slot, int row) {
    float top = -INFINITY;
#pragma unroll
    for (int k = 0; k < 4; ++k) top = fmaxf(top, stat_at(u, k, row)[0]);
    const float2 pt = stat_partial(fold(u, row, top));
    unsigned long long* const to = tagged_words(slot, row) + rank * R;
    put_word(to, tagged(pt.x, tag0 + u));
    put_word(to + kEntWords, tagged(pt.y, tag0 + u));
  };

  // Summed: the row's common reference in unit u of this team.  A slot is used again kRefSlots units later: who
  // finds the references of unit v has published unit v - kRefAhead, so every CTA is done with the
  // units before v - kRefAhead - 2 kResRing + 1.
  auto ref_word = [&](unsigned u, int row) {
    return p.xch + 2 * (size_t)kXchPairs + (size_t)(team * kRefSlots + (int)(u % kRefSlots)) * R + row;
  };
  // Waits for it; `word` was read before.  Whoever has it finds the row's summed words clean.
  auto have_ref = [&](unsigned u, int row, unsigned long long& word) {
    for (long long t0 = 0; !__all_sync(0xffffffffu, word_has(word, tag0 + u));) {
      if (!__all_sync(0xffffffffu, keep_polling(t0))) return false;
      word = get_word_acquire(ref_word(u, row));
    }
    return true;
  };

  if (warp == kResWarps) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      const uint64_t pol_keep = l2_policy_evict_last(), pol_stream = l2_policy_evict_first();
      unsigned kt = 0, qn = 0;                             // K tiles, Q blocks loaded so far
      bool ok = true;
      for (Walk w = walk_from(); w.pi < n_prob && ok; walk_on(w)) {
        const ResShare s = prob_s[w.pi];
        const CUtensorMap* map_k = &p.map_k[w.pi];
        for (int a = 0; a < s.c && ok; a += 4) {
          const int sg = kt % kStages, n = min(4, s.c - a);
          ok = mbar_wait_producer(bar(L::kKEmpty + sg), ((kt / kStages) & 1u) ^ 1u, abort_flag, kWaitCycles);
          if (!ok) break;
          mbar_expect_tx(bar(L::kKFull + sg), n * kResChunk * D * 2);
          // the last chunk may reach beyond the sequence (into zero fill): the causal mask discards those keys
          for (int q = 0; q < n; ++q)
            for (int c = 0; c < L::kSub; ++c)
              tma_load_3d_hint(base + sg * L::kTile + c * L::kTileSub + q * (kResChunk * 128), map_k, bar(L::kKFull + sg),
                               c * 64, (s.lo + a + q) * kResChunk, w.g, pol_stream);
          ++kt;
          if (a > 0) continue;
          ok = mbar_wait_producer(bar(L::kQEmpty + (qn & 1)), ((qn >> 1) & 1u) ^ 1u, abort_flag, kWaitCycles);
          if (!ok) break;
          mbar_expect_tx(bar(L::kQFull + (qn & 1)), L::kQ);
          for (int c = 0; c < L::kSub; ++c)
            tma_load_3d_hint(base + L::kQOff + (qn & 1) * L::kQ + c * L::kQSub, &p.map_q[w.pi], bar(L::kQFull + (qn & 1)),
                             c * 64, 0, w.g * p.group, pol_keep);
          ++qn;
        }
      }
      // every copy this thread issued must have landed before the CTA may exit
      for (unsigned i = qn > 2 ? qn - 2 : 0; i < qn; ++i) mbar_drain(bar(L::kQFull + (i & 1)), (i >> 1) & 1u, abort_flag);
      for (unsigned i = kt > kStages ? kt - kStages : 0; i < kt; ++i)
        mbar_drain(bar(L::kKFull + i % kStages), (i / kStages) & 1u, abort_flag);
    }
  } else if (warp == kResWarps + 1) {
    // ---------------- MMA issuer ----------------
    if (lane == 0) {
      const uint64_t q_desc0 = smem_desc(base + L::kQOff), k_desc0 = smem_desc(base);
      unsigned kt = 0, qn = 0;                             // K tiles, Q blocks so far
      bool ok = true;
      auto wait = [&](int b, unsigned parity) { return mbar_wait_producer(bar(b), parity, abort_flag, kWaitCycles); };
      for (Walk w = walk_from(); w.pi < n_prob && ok; walk_on(w)) {
        const int c = prob_s[w.pi].c;
        const uint32_t idesc = instr_desc(128, R) | (prob_s[w.pi].p.negate ? 1u << 13 : 0u);
        if (c == 0) continue;
        if (!(ok = wait(L::kQFull + (qn & 1), (qn >> 1) & 1u))) break;
        const uint64_t qd = q_desc0 + (uint64_t)(((qn & 1) * L::kQ) >> 4);
        for (int a = 0; a < c; a += 4, ++kt) {
          const unsigned sg = kt % kStages, slot = kt % kSlots;
          if (!(ok = wait(L::kKFull + sg, (kt / kStages) & 1u))) break;
          if (!(ok = wait(L::kFree + slot, ((kt / kSlots) & 1u) ^ 1u))) break;
          tc_fence_after();
          const uint64_t kd = k_desc0 + (uint64_t)((sg * L::kTile) >> 4);
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk) {
            const uint32_t ko = (kk / 4) * L::kTileSub + (kk % 4) * 32, qo = (kk / 4) * L::kQSub + (kk % 4) * 32;
            tc_mma_bf16(tmem + slot * R, kd + (ko >> 4), qd + (qo >> 4), idesc, kk > 0);
          }
          fl->mma_in_flight = 1;
          tc_commit(bar(L::kKEmpty + sg));                 // K stage reusable once these MMAs have read it
          tc_commit(bar(L::kFull + slot));                 // logits ready for the compute warps
        }
        if (!ok) break;
        tc_commit(bar(L::kQEmpty + (qn & 1)));
        ++qn;
      }
      // all issued MMAs must retire before tensor memory is freed
      if (fl->mma_in_flight) {
        tc_commit(bar(L::kDrain));
        if (mbar_drain(bar(L::kDrain), 0, abort_flag)) fl->mma_in_flight = 0;
      }
    }
  } else if (warp == kResWarps + 3) {
    // ---------------- this CTA's statistics ----------------
    const int row = lane;
    // Common references of a unit (a row's largest logit over the first four keys and the last four that all of its rows
    // see) and clean summed words: 32 rows by 8 keys, two m16n8 products.  Which of a thread's eight consecutive elements
    // stands for which k of the instruction does not matter as long as both operands agree.  (Unrolled over both halves of the
    // rows it cost every form: 28 layers of 5003 keys, direct, 3.83 us a layer, so 3.74; rolled up altogether, with one load
    // in flight, a layer of one KV head and 40000 keys 18.8 -> 20.9.)
    auto find_refs = [&](unsigned v) {
      const int gu = team + (int)v * teams, pi = gu / n_kv, g = gu - pi * n_kv;
      if (pi >= n_prob) return;
      __syncwarp();                                        // the products want the whole warp
      const ResProblem& pb = prob_s[pi].p;
      const int open = pb.n_keys - p.window, t = lane & 3, n = lane >> 2;
      const int key = n < 4 ? min(n, open) : max(0, open - (n - 4));
      const __nv_bfloat16* const k = pb.k + g * p.k_stride_head + key * p.k_stride_token + t * 8;
      float ref = 0.f;
#pragma unroll 1
      for (int m = 0; m < 2; ++m) {
        const __nv_bfloat16* q[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int r = m * 16 + h * 8 + n, at = is_row(r) ? r / p.w_pad * p.window + (r & (p.w_pad - 1)) : 0;
          q[h] = pb.q + ((size_t)g * p.group * p.window + at) * D + t * 8;
        }
        float acc[4] = {};
#pragma unroll
        for (int c = 0; c < D; c += 32) {
          const uint4 a = __ldg(reinterpret_cast<const uint4*>(q[0] + c)), b = __ldg(reinterpret_cast<const uint4*>(q[1] + c));
          const uint4 x = __ldg(reinterpret_cast<const uint4*>(k + c));
          mma_16x8x16(acc, a.x, b.x, a.y, b.y, x.x, x.y);
          mma_16x8x16(acc, a.z, b.z, a.w, b.w, x.z, x.w);
        }
        const float c2 = pb.negate ? -pb.c2 : pb.c2;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float x = fmaxf(acc[2 * h] * c2, acc[2 * h + 1] * c2);
          x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 1));
          x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 2));
          x = __shfl_sync(0xffffffffu, x, (row & 7) * 4);
          if (row >> 3 == 2 * m + h) ref = x;
        }
      }
      if (!is_row(row) || !(fabsf(ref) < 3.0e38f)) ref = 0.f;
      reinterpret_cast<ulonglong2*>(p.sums)[(size_t)gu * R + row] = make_ulonglong2(0, 0);
      __threadfence();
      put_word(ref_word(v, row), tagged(ref, tag0 + v));
    };
    unsigned u = 0;
    int slot = 0;
    unsigned long long ref = 0;
    if (p.sums && rank < kRefAhead) find_refs(rank);
    for (Walk w = walk_from(); w.pi < n_prob; walk_on(w), ++u) {
      const size_t at = (size_t)unit_of(w) * R + row;
      if (p.sums && !have_ref(u, row, ref)) break;
      if (!__all_sync(0xffffffffu, mbar_wait(bar(L::kStats + (int)(u % kResRing)), (u / kResRing) & 1u, abort_flag))) break;
      if (!p.sums) {
        publish(u, slot, row);
        slot = next_slot(slot);
      } else if (is_row(row)) {
        const RowStat f = fold(u, row, word_value(ref));
        unsigned long long* const to = p.sums + 2 * at;
        const bool fits = f.Z < kSumLimit && fabsf(f.U) < kSumLimit;
        if (!fits) atomicOr(to, kSumOver);
        atomicAdd(to, kSumCount + (fits ? (unsigned long long)__float2ll_rn(f.Z * kSumUnit) : 0ull));
        atomicAdd(to + 1, kSumCount + kSumBias + (fits ? (unsigned long long)__float2ll_rn(f.U * kSumUnit) : 0ull));
      }
      if (p.sums) {
        if ((u + kRefAhead) % (unsigned)G == (unsigned)rank) find_refs(u + kRefAhead);
        ref = get_word_acquire(ref_word(u + 1, row));
      }
    }
  } else if (warp == kResWarps + 2) {
    // ---------------- normalisers ----------------
    const int row = lane;
    const bool valid = is_row(row);
    unsigned u = 0;
    int slot = 0;
    unsigned long long ref = 0;
    bool live = true;
    // A row's word once all CTAs are in it (rows that exist), or the CTA gives up.
    auto summed = [&](const unsigned long long* at) {
      unsigned long long x = 0;
      for (long long t0 = 0;;) {
        if (valid) x = get_word(at);
        if (__all_sync(0xffffffffu, !valid || (int)(x >> 56) == G)) break;
        if (!__all_sync(0xffffffffu, keep_polling(t0))) { live = false; break; }
      }
      return x;
    };
    for (Walk w = walk_from(); w.pi < n_prob; walk_on(w), ++u, slot = next_slot(slot)) {
      const bool leaves = (int)(u % (unsigned)G) == rank;  // one CTA of the team leaves the rows' entropies
      const unsigned long long* const words = tagged_words(slot, row);
      const size_t at = (size_t)unit_of(w) * R + row;
      const unsigned tag = tag0 + u;
      float lse = -INFINITY, Z = 0.f, log_z = 0.f;
      bool direct = p.sums == nullptr;
      if (!direct) {
        if (!have_ref(u, row, ref)) break;
        const unsigned long long x = summed(p.sums + 2 * at);
        if (!live) break;
        Z = (float)(x & (kSumOver - 1)) * (1.f / kSumUnit);
        log_z = log2f(Z);                                  // Z is some tens: the fast one errs as much as lse's last bit
        lse = word_value(ref) + log_z;
        ref = get_word_acquire(ref_word(u + 1, row));
        if (__any_sync(0xffffffffu, (x & kSumOver) != 0)) {   // the same answer in every CTA
          direct = true;
          __threadfence_block();
          publish(u, slot, row);
        }
      }
      if (direct) {
        constexpr int kAt = 20;                            // words in flight
        float M = -INFINITY, Ws = 0.f;
        long long t0 = 0;
        for (int s0 = 0; s0 < G && live; s0 += kAt) {
          float l[kAt];
          for (;;) {
            bool all = true;
#pragma unroll
            for (int i = 0; i < kAt; ++i) {
              unsigned long long x = 0;
              if (s0 + i < G) x = get_word(words + (s0 + i) * R);
              l[i] = s0 + i < G ? word_value(x) : -INFINITY;
              all = all && (s0 + i >= G || word_has(x, tag));
            }
            if (__all_sync(0xffffffffu, all)) break;
            if (!__all_sync(0xffffffffu, keep_polling(t0))) { live = false; break; }
          }
          float top = M;
#pragma unroll
          for (int i = 0; i < kAt; ++i) top = fmaxf(top, l[i]);
          if (top == -INFINITY) continue;
          Ws *= M == -INFINITY ? 0.f : fast_exp2(M - top);
#pragma unroll
          for (int i = 0; i < kAt; ++i) Ws += l[i] == -INFINITY ? 0.f : fast_exp2(l[i] - top);
          M = top;
        }
        if (!live) break;
        lse = Ws > 0.f ? M + __log2f(Ws) : -INFINITY;
      }
      lse_s[u % kResRing * R + row] = valid && lse != -INFINITY ? -lse : -INFINITY;
      __threadfence_block();
      __syncwarp();
      if (lane == 0) fl->known = (int)u + 1;
      if (!leaves) continue;
      float ent = 0.f;
      if (!direct) {
        const unsigned long long x = summed(p.sums + 2 * at + 1);
        if (!live) break;
        const long long us = (long long)(x & (kSumCount - 1)) - (long long)(kSumBias * (unsigned long long)G);
        ent = kLn2 * (log_z - (float)us * (1.f / kSumUnit) / Z);
      } else {
        constexpr int kAt = 10;
        long long t0 = 0;
        for (int s0 = 0; s0 < G && live; s0 += kAt) {
          unsigned long long l[kAt], h[kAt];
          for (;;) {
            bool all = true;
#pragma unroll
            for (int i = 0; i < kAt; ++i) {
              const int from = min(s0 + i, G - 1);
              l[i] = get_word(words + from * R);
              h[i] = get_word(words + from * R + kEntWords);
            }
#pragma unroll
            for (int i = 0; i < kAt; ++i) all = all && word_has(h[i], tag);
            if (__all_sync(0xffffffffu, all)) break;
            if (!__all_sync(0xffffffffu, keep_polling(t0))) { live = false; break; }
          }
#pragma unroll
          for (int i = 0; i < kAt; ++i) {
            const float lv = word_value(l[i]);
            if (s0 + i < G && lv != -INFINITY) ent = fmaf(fast_exp2(lv - lse), word_value(h[i]) + (lse - lv), ent);
          }
        }
        if (!live) break;
        ent = lse != -INFINITY ? kLn2 * ent : 0.f;
      }
      for (int r = row; r < kRowBlock; r += R) p.row_ent[(size_t)unit_of(w) * kRowBlock + r] = r == row && valid ? ent : 0.f;
    }
  } else {
    // ---------------- statistics and column sums ----------------
    // Lane = key, RT rows per thread; T tiles' loads travel together.
    constexpr int RT = R / kResSubs, T = 4, kLanes = 32 / RT;
    const int quarter = warp & 3, sub = warp >> 2, set0 = sub * RT;
    const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
    const float inv_w = 1.0f / (float)p.window;
    auto slot_addr = [&](unsigned tile) { return lane_base + tile % kSlots * R; };
    auto full = [&](unsigned tile) {                       // the MMAs have left a tile's logits
      uint32_t ok;
      asm volatile("{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
                   : "=r"(ok) : "r"(bar(L::kFull + (int)(tile % kSlots))), "r"((tile / kSlots) & 1u) : "memory");
      return __all_sync(0xffffffffu, ok) != 0;
    };
    // Where the statistics (e) and the column sums (s) are: unit, its first tile, tiles.
    struct At { Walk w; unsigned u, tile; };
    auto tiles_of = [&](const At& a) { return (prob_s[a.w.pi].c + 3) / 4; };
    auto next_unit = [&](At& a) {
      a.tile += tiles_of(a);
      ++a.u;
      walk_on(a.w);
    };
    At e{walk_from(), 0, 0}, s = e;
    // The common references of this warp's rows in unit e (summed; lane l holds that of row l % RT), first looked for
    // a unit ahead.
    auto look_for_refs = [&](unsigned u) { return p.sums ? get_word(ref_word(u, set0 + lane % RT)) : 0ull; };
    unsigned long long refs = look_for_refs(0);
    auto have_refs = [&]() {
      if (!p.sums || __all_sync(0xffffffffu, word_has(refs, tag0 + e.u))) return true;
      refs = look_for_refs(e.u);
      return __all_sync(0xffffffffu, word_has(refs, tag0 + e.u)) != 0;
    };
    long long t0 = 0;
    while (s.w.pi < n_prob) {
      if (__all_sync(0xffffffffu, fl->known > (int)s.u)) {
        // ---- column sums: this warp takes every fourth tile, all rows ----
        __threadfence_block();
        t0 = 0;
        const ResShare& sh = prob_s[s.w.pi];
        const uint64_t c22 = pack2(sh.p.c2, sh.p.c2);
        const int last_open_key = sh.p.n_keys - p.window;  // the last key every window row sees
        const float* const nlse = lse_s + s.u % kResRing * R;
        for (int i = (sub + s.u) % kResSubs; i < tiles_of(s); i += kResSubs) {
          const int j = (sh.lo + 4 * i) * kResChunk + quarter * 32 + lane, hi = min((sh.lo + sh.c) * kResChunk, sh.p.n_keys);
          const int i_min = j - last_open_key;             // window rows below do not see key j
          const bool plain = __all_sync(0xffffffffu, i_min <= 0);
          float* const out = sh.p.cols + (size_t)(s.w.g * p.group) * p.col_stride + j;
          float tot = 0.f, v[R];
          int head = 0;
          tc_fence_after();
          tmem_ld(slot_addr(s.tile + i), v);
          if (!plain) {
#pragma unroll
            for (int x = 0; x < R; ++x)
              if ((x & (p.w_pad - 1)) < i_min) v[x] = kMaskedAcc;
          }
#pragma unroll
          for (int k = 0; k < R / 8; ++k) {
            uint64_t s2 = pack2(0.f, 0.f);
#pragma unroll
            for (int x = 8 * k; x < 8 * k + 8; x += 4) {
              const float4 n4 = *reinterpret_cast<const float4*>(nlse + x);
              s2 = add2(s2, exp2_sfu2(fma2(pack2(v[x], v[x + 1]), c22, pack2(n4.x, n4.y))));
              s2 = add2(s2, exp2_sfu2(fma2(pack2(v[x + 2], v[x + 3]), c22, pack2(n4.z, n4.w))));
            }
            float lo, up;
            unpack2(s2, lo, up);
            tot += lo + up;
            if (((8 * k + 8) & (p.w_pad - 1)) == 0) {
              if (head < p.group && j < hi) out[(size_t)head * p.col_stride] = tot * inv_w;
              ++head;
              tot = 0.f;
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(L::kFree + (int)((s.tile + i) % kSlots)));   // the next MMA may write it
        }
        if (lane == 0) {
          int* const ctr = &flags->sum_ctr[s.u % kResRing];
          __threadfence_block();
          if (atomicAdd(ctr, 1) == kResWarps - 1) {
            *ctr = 0;
            __threadfence_block();
            fl->summed = (int)s.u + 1;
          }
        }
        __syncwarp();
        next_unit(s);
        continue;
      }
      // ---- statistics of the next unit: all of its tiles and references are there, and a place for its statistics is ----
      if (e.w.pi < n_prob && __all_sync(0xffffffffu, fl->summed + kResRing > (int)e.u) && full(e.tile + tiles_of(e) - 1) && have_refs()) {
        t0 = 0;
        tc_fence_after();
        const ResShare& sh = prob_s[e.w.pi];
        const float c2 = sh.p.c2;
        const uint64_t c22 = pack2(c2, c2);
        const int last_open_key = sh.p.n_keys - p.window, hi = (sh.lo + sh.c) * kResChunk;
        const float masked = fmaxf(__fdividef(kMasked, c2), kMaskedAcc);   // times c2: finite, and 2^x flushes to 0
        const float common = word_value(refs);
        refs = look_for_refs(e.u + 1);
        const int tiles = tiles_of(e), j0 = sh.lo * kResChunk + quarter * 32 + lane;
        float v[T * RT];
        // The logits of tiles [i0, i0 + n_here), where a row does not see a key: masked.
        auto load = [&](int i0, int n_here) {
#pragma unroll
          for (int k = 0; k < T; ++k) tmem_ld_issue<RT>(slot_addr(e.tile + i0 + min(k, n_here - 1)) + set0, v + k * RT);
          tmem_ld_wait(v);
#pragma unroll
          for (int k = 0; k < T; ++k) {
            const int jt = (sh.lo + 4 * (i0 + k)) * kResChunk;
            if (k >= n_here || (jt + kKeyTile <= hi && jt + kKeyTile - 1 <= last_open_key)) continue;
            const int j = j0 + (i0 + k) * kKeyTile, over = j < hi ? j - last_open_key : 0x7fffffff;
#pragma unroll
            for (int x = 0; x < RT; ++x)               // rows i < over do not see this key
              if (((set0 + x) & (p.w_pad - 1)) < over) v[k * RT + x] = masked;
          }
        };
        // Moves the references to the largest logits of the loaded tiles where these are larger.
        uint64_t nref2[RT / 2], Z2[RT / 2], U2[RT / 2];  // pairs of rows: -reference, Z, U
        auto raise_refs = [&](int n_here) {
#pragma unroll
          for (int k = 0; k < RT / 2; ++k) {
            float m[2], r[2];
            unpack2(nref2[k], r[0], r[1]);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              m[h] = v[2 * k + h];
#pragma unroll
              for (int x = 1; x < T; ++x)
                if (x < n_here) m[h] = fmaxf(m[h], v[x * RT + 2 * k + h]);
              m[h] = warp_max(m[h]) * c2;
              if (m[h] > 0.5f * masked * c2) r[h] = fminf(r[h], -m[h]);
            }
            nref2[k] = pack2(r[0], r[1]);
          }
        };
#pragma unroll
        for (int k = 0; k < RT / 2; ++k)
          nref2[k] = pack2(-__shfl_sync(0xffffffffu, common, 2 * k), -__shfl_sync(0xffffffffu, common, 2 * k + 1));
        // At first with the team's references, or the first tile's largest logits; where logits tower over these, once
        // more with the largest of all (they are still there).
        for (int attempt = 0; attempt < 2; ++attempt) {
          const bool scan = attempt > 0;
          if (scan) {
            for (int i0 = 0; i0 < tiles; i0 += T) {
              load(i0, min(T, tiles - i0));
              raise_refs(min(T, tiles - i0));
            }
          }
#pragma unroll
          for (int k = 0; k < RT / 2; ++k) Z2[k] = U2[k] = 0;
          for (int i0 = 0; i0 < tiles; i0 += T) {
            const int n_here = min(T, tiles - i0);
            load(i0, n_here);
            if (!p.sums && !scan && i0 == 0) {
#pragma unroll
              for (int k = 0; k < RT / 2; ++k) nref2[k] = pack2(INFINITY, INFINITY);
              raise_refs(1);
#pragma unroll
              for (int k = 0; k < RT / 2; ++k) {
                float r0, r1;
                unpack2(nref2[k], r0, r1);
                nref2[k] = pack2(r0 == INFINITY ? 0.f : r0, r1 == INFINITY ? 0.f : r1);
              }
            }
#pragma unroll
            for (int y = 0; y < T; ++y) {
              if (y >= n_here) break;
#pragma unroll
              for (int k = 0; k < RT / 2; ++k) {
                const uint64_t x2 = fma2(pack2(v[y * RT + 2 * k], v[y * RT + 2 * k + 1]), c22, nref2[k]), p2 = exp2_sfu2(x2);
                Z2[k] = add2(Z2[k], p2);
                U2[k] = fma2(p2, x2, U2[k]);
              }
            }
          }
          float most = 0.f;
#pragma unroll
          for (int k = 0; k < RT / 2; ++k) {
            float a, b;
            unpack2(Z2[k], a, b);
            most = fmaxf(most, fmaxf(a, b));
          }
          if (!__any_sync(0xffffffffu, most > 1.0e18f)) break;
        }
        tc_fence_before();
        float ref[RT], Z[RT], U[RT];
#pragma unroll
        for (int k = 0; k < RT / 2; ++k) {
          unpack2(nref2[k], ref[2 * k], ref[2 * k + 1]);
          unpack2(Z2[k], Z[2 * k], Z[2 * k + 1]);
          unpack2(U2[k], U[2 * k], U[2 * k + 1]);
        }
        const float ref_l = -lane_element(ref, lane), Z_l = warp_sum_scatter(Z, lane), U_l = warp_sum_scatter(U, lane);
        if (lane % kLanes == 0) {
          float* const st = stat_at(e.u, quarter, set0 + lane / kLanes);
          st[0] = p.sums || Z_l != 0.f ? ref_l : -INFINITY;
          st[1] = Z_l;
          st[2] = U_l;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(L::kStats + (int)(e.u % kResRing)));
        next_unit(e);
        continue;
      }
      // nothing to do yet
      if (!__all_sync(0xffffffffu, keep_polling(t0))) break;
      __nanosleep(20);
    }
  }

  // ---------------- teardown ----------------
  tc_fence_before();
  __syncthreads();
  if (*abort_flag && threadIdx.x == 0) atomicCAS(p.status, 0, (int)STRUCTKV_ERR_TIMEOUT);
  // tensor memory is freed only when no MMA of this CTA can still write to it
  if (warp == kResWarps + 1 && !fl->mma_in_flight) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
  if (threadIdx.x == 0) fl->last = atomicAdd(p.ctl + kCtlExit, 1) == (int)gridDim.x - 1;
  __syncthreads();
  if (fl->last) pass_tags_on(p.xch, p.ctl, tag0 - 1u + (unsigned)((n_prob * n_kv + teams - 1) / teams), (int)threadIdx.x, (int)blockDim.x);
}

template <int D, int MAXP>
cudaError_t res_launch(const ResParams<MAXP>& p, int device, cudaStream_t st) {
  auto kern = tc_resident<D, MAXP>;
  constexpr int kAlloc = ResSmem<D, MAXP>::kAlloc;
  static std::atomic<unsigned long long> ready{0};        // devices whose shared-memory limit has been raised
  const unsigned long long bit = 1ull << (device & 63);
  if (!(ready.load(std::memory_order_acquire) & bit)) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kAlloc);
    if (e != cudaSuccess) return e;
    ready.fetch_or(bit, std::memory_order_release);
  }
  return launch_cooperative(kern, dim3(p.team * p.teams), dim3(kResThreads), kAlloc, st, p);
}
#endif  // __CUDACC__

// One translation unit per head dimension instantiates the kernels.
cudaError_t res_launch_64(const ResParams<1>& p, int device, cudaStream_t st);
cudaError_t res_launch_64(const ResParams<kMaxBatch>& p, int device, cudaStream_t st);
cudaError_t res_launch_128(const ResParams<1>& p, int device, cudaStream_t st);
cudaError_t res_launch_128(const ResParams<kMaxBatch>& p, int device, cudaStream_t st);

}  // namespace skv
