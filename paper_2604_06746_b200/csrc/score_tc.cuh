// Tensor-core scorer for bf16 storage on sm_100a: TMA-staged K tiles, tcgen05.mma with fp32
// accumulators in tensor memory, softmax statistics / column sums computed straight out of
// tensor memory.  ONE persistent kernel runs both passes over every problem of a call (a layer, or
// a sequence of a packed batch):
//
//   pass 1  per score row the softmax statistics (ref, Z, U) over a key range
//   pass 2  per head the column sums of exp(x - lse) for every key
//
// A task is (pass, problem, unit, key range); a unit is (KV group, block of up to 256 score rows).
// CTAs (one per SM) draw tasks in order from one ticket counter.  A pass-2 task waits until all
// pass-1 tasks of its unit are stored and merged; those have smaller tickets, so every one of
// them has been drawn by a CTA that is running, and works on nothing that waits for a larger
// ticket: the waits end whatever the number of resident CTAs.  Neighbouring layers interleave
// (P1(0), P1(1), P2(0), P1(2), P2(1), ...), so a unit's statistics are ready long before its second
// pass is drawn, no SM idles while the slowest CTA of a pass finishes, and nothing of a CTA's set-up
// (launch, tensor-memory allocation, first copies) is paid per layer: with two launches per layer
// that set-up and the uneven last wave were 12 % of a layer of 131072 keys and a third at 32768.
// Which keys a partial of pass 1 covers (a segment) depends on the shape alone, so results depend neither on
// timing nor on how many segments a task runs.
//
// Two layouts of the score rows:
//   wide    (more than 64 rows per KV group) pass 1 D[rows, keys] = Q K^T, lane = row; pass 2
//           D[keys, rows] = K Q^T, lane = key: both reductions are loops inside one thread.  Both
//           issue M128 x N256 MMAs: pass 1 one 128-row half of Q with a PAIR of key tiles (two
//           neighbouring stages of the K ring form one operand), pass 2 one key tile with the whole
//           256-row block.
//   narrow  (at most 64 rows per KV group, e.g. 4 heads x a window of 8) D[keys, rows] in both passes,
//           N = 32 or 64: in the wide layout three quarters of the lanes would hold padding.  Pass 1
//           keeps its statistics per (lane, row) and folds the lanes once per task.  The path is then
//           bound by reading K (on the CUDA cores it took 25 times as long at 32768 keys, window 8).
// A head's window rows are padded to the next power of two (8 at least); the tensor map fills the
// padding with zeros and the statistics mark it invalid.
//
// What bounds the wide layout: the exponentials.  2 x H w N of them at 16 per clock and SM (plus what
// the FMA pipe takes over), and, since both pipes and the tensor cores are then busy together, the
// power cap: at 131072 keys the clock settles near 1.6 GHz.
//
// Warp roles: warp 0 = ticket taker and TMA producer, warp 1 = MMA issuer (owns the tensor-memory
// allocation), warp 2 = hands a unit's log-sum-exps to pass 2, warp 3 = counts finished
// pass-1 tasks (the CTA whose task completes a unit merges its partials), warps 4-19 = compute (four
// per scheduler).  Tasks reach the consumers through a ring of descriptors in shared memory that holds
// all they need (indexing the launch's parameters by problem cost 1500 clocks of constant-cache misses
// a task).
// Every wait is bounded; on expiry the CTA records STRUCTKV_ERR_TIMEOUT and stops issuing work;
// it then waits (with a fresh bound that ignores the abort flag) for its own copies and MMAs in
// flight, and frees tensor memory only if those MMAs are known to have retired.
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>

#include <atomic>

#include "common.cuh"

namespace skv {

constexpr int kStages = 4;             // K tile ring
constexpr int kTaskRing = 4;           // task descriptors in flight inside a CTA
constexpr int kHelperWarps = 4;
constexpr int kComputeWarps = 16;
constexpr int kTcThreads = (kHelperWarps + kComputeWarps) * 32;   // 20 warps: the most that fit at 96 registers a thread
constexpr float kMasked = -1.0e30f;    // exponent standing for -inf: 2^x flushes to 0 and 0 * x stays finite
constexpr float kMaskedAcc = -3.0e38f; // the same for an accumulator, before the scaling by c2 >= 1e-30
constexpr int kFullWeight = 20;        // weight of a full row block when key ranges are dealt out (see tc_deal)

// What the kernel is compiled for.  kHurry: pass 2 has nothing to do but wait for pass 1 (one layer, a batch), so the compute
// warps count their arrivals and merge the row statistics themselves, a thread per row, instead of leaving it to one helper
// warp beside them (at 8192 keys 2 us instead of 6).  With layers to interleave the helpers' time is hidden and the compute
// warps' is not (32 layers of 5003 keys, when both were one kernel and a pass slower than now: 317 us in a hurry, 300
// without).  Then 32 layers of 1500 keys took 117.7 us instead of 115.5, one layer of 9300 33.9 instead of 33.6.
// kBrief: pass 2's arithmetic in one copy instead of two.  Short tasks alternate with pass 1 and are as long as it takes to fetch
// them; long ones gain by a second load under way earlier.  us, two copies / one: window 64, 32 layers of 1500 keys 115.5 /
// 109.6, of 5003 262 / 246, of 8192 387 / 370, 16 of 16384 366 / 356, of 24000 491 / 491, of 32768 657 / 657, 8 of 65536 656 /
// 690; window 128, 28 query heads over 4 KV heads, 16 of 5000 278 / 267, 12 of 10000 372 / 355, 8 of 20000 398 / 408; a layer
// by itself, 9300 keys 33.6 / 35.2, 131072 164 / 170.
enum TcForm { kAmong = 0, kBrief, kHurry };
// (KV group, row block, pair of key tiles) triples of a layer up to which its tasks count as short.
constexpr int kBriefPairs = 768;

// Layout classes of the kernel (template argument).
enum TcShape { kWide16 = 0, kWide32, kWide64, kWide128, kWide256, kNarrow32, kNarrow64 };

// One independent scoring problem of a launch: a layer, or a sequence of a packed batch.
struct TcProblem {
  float* cols;                         // pass-2 output of head 0, key 0
  int key0, n_keys;                    // rows of the K tensor
  int map, head0;                      // tensor maps; first head in the Q tensor
  float c2, inv_c2, v_min;             // |scale| * log2(e), at least 1e-30; 1 / c2; -125 / c2
  int negate;                          // the scale is negative: the MMA negates its A operand
  int s1, t1, t2, part0;               // key segments of pass 1, tasks of the two passes; first partial of pass 1
};
// A run of consecutive tickets, from `first` on: the tasks of one pass of one problem.
struct TcPhase { int first; unsigned char prob, pass; };

template <int MAXP>
struct alignas(64) TcParams {
  CUtensorMap map_q[MAXP], map_k[MAXP];
  TcProblem prob[MAXP];
  TcPhase phase[4 * MAXP + 1];         // the last one only carries the ticket count
  int n_phase, n_prob;
  int window, w_pad, group, rows_pg, n_rb, n_units;    // w_pad: rows a head occupies; rows_pg = group * w_pad
  int w_shift;                         // log2(w_pad)
  int w_group, w_total, w_last;        // weights of a KV group, of all, of a group's last row block
  int* ctl;                            // ticket, exits; then arrivals and ready flags [kMaxBatch][kQueueUnits]
  float2* part;                        // [pass-1 task][256] (log-sum-exp, entropy) in bits
  float* nlse;                         // [problem][unit][256] -log2-sum-exp of a row (-inf: no row)
  float* row_ent;                      // [problem][unit][256] entropy of a row, nats (0: no row)
  long long col_stride;
  int* status;
  int form;                            // TcForm
};
constexpr int kCtlTicket = 0, kCtlArrive = 64, kCtlReady = 64 + kMaxBatch * kQueueUnits;
static_assert(kCtlInts == 64 + 2 * kMaxBatch * kQueueUnits, "control block");

// Tasks of a problem are dealt out to its units in proportion to their weights: unit u owns tasks
// [tc_deal(W(u)), tc_deal(W(u + 1))), W = sum of the weights before it.  A group's last row block that
// holds a single 128-row half costs half a full one per key in pass 1 and between a half and three
// quarters in pass 2: weight 13 of 20.
__host__ __device__ inline int tc_deal(int w_before, int tasks, int w_total) { return w_before * tasks / w_total; }

#ifdef __CUDACC__

// ---- PTX wrappers ----------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\n"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// Same test, letting the hardware suspend the thread for up to kSuspendNs while the phase
// is incomplete: a waiting producer then issues (almost) no instructions on its scheduler.
constexpr uint32_t kSuspendNs = 1000;
__device__ __forceinline__ bool mbar_try_suspend(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\n"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
      "selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok) : "r"(bar), "r"(parity), "r"(kSuspendNs) : "memory");
  return ok != 0;
}
// Bounded wait of a producer (TMA / MMA warp): long, rarely latency critical.
__device__ __forceinline__ bool mbar_wait_producer(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                                   unsigned long long limit) {
  if (mbar_try(bar, parity)) return true;
  const long long t0 = clock64();
  for (;;) {
#pragma unroll 1
    for (int i = 0; i < 16; ++i)
      if (mbar_try_suspend(bar, parity)) return true;
    if (*abort_flag) return false;
    if ((unsigned long long)(clock64() - t0) > limit) { *abort_flag = 1; return false; }
  }
}
// Bounded wait.  Returns false if the barrier did not flip within `limit` cycles or the CTA is
// aborting; the first waiter whose bound expires raises the CTA's abort flag.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                          unsigned long long limit = kWaitCycles) {
  if (mbar_try(bar, parity)) return true;
  const long long t0 = clock64();
  for (;;) {
#pragma unroll 1
    for (int i = 0; i < 256; ++i)
      if (mbar_try(bar, parity)) return true;
    if (*abort_flag) return false;
    if ((unsigned long long)(clock64() - t0) > limit) { *abort_flag = 1; return false; }
  }
}
// Bounded wait for work this thread itself put in flight (copies, MMAs): runs after an abort as
// well, so it ignores the abort flag and starts its own timer.  False = still in flight.
__device__ __forceinline__ bool mbar_drain(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                           unsigned long long limit = kWaitCycles) {
  if (mbar_try(bar, parity)) return true;
  const long long t0 = clock64();
  for (;;) {
#pragma unroll 1
    for (int i = 0; i < 256; ++i)
      if (mbar_try(bar, parity)) return true;
    if ((unsigned long long)(clock64() - t0) > limit) { *abort_flag = 1; return false; }
  }
}
// d[16 x 8] += a[16 x 16] b[16 x 8], for products too small for a tcgen05 tile.
__device__ __forceinline__ void mma_16x8x16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// 3-D tile copy with an L2 eviction-priority hint for the lines it brings in.
__device__ __forceinline__ void tma_load_3d_hint(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0,
                                                 int c1, int c2, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
      "[%0], [%1, {%3, %4, %5}], [%2], %6;"
      ::"r"(dst), "l"((uint64_t)map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "l"(policy) : "memory");
}
__device__ __forceinline__ uint64_t l2_policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t l2_policy_evict_normal() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t l2_policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// 32 lanes x N consecutive fp32 columns: thread l of the warp receives row (lane base + l).  The
// loaded registers are operands of the wait, so no use of them can be scheduled ahead of it.
__device__ __forceinline__ void tmem_ld(uint32_t taddr, float (&v)[32]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
               "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]),
                 "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15]),
                 "=f"(v[16]), "=f"(v[17]), "=f"(v[18]), "=f"(v[19]), "=f"(v[20]), "=f"(v[21]), "=f"(v[22]),
                 "=f"(v[23]), "=f"(v[24]), "=f"(v[25]), "=f"(v[26]), "=f"(v[27]), "=f"(v[28]), "=f"(v[29]),
                 "=f"(v[30]), "=f"(v[31])
               : "r"(taddr) : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]),
                 "+f"(v[8]), "+f"(v[9]), "+f"(v[10]), "+f"(v[11]), "+f"(v[12]), "+f"(v[13]), "+f"(v[14]), "+f"(v[15]),
                 "+f"(v[16]), "+f"(v[17]), "+f"(v[18]), "+f"(v[19]), "+f"(v[20]), "+f"(v[21]), "+f"(v[22]),
                 "+f"(v[23]), "+f"(v[24]), "+f"(v[25]), "+f"(v[26]), "+f"(v[27]), "+f"(v[28]), "+f"(v[29]),
                 "+f"(v[30]), "+f"(v[31])
               :: "memory");
}
// The load and its wait apart: several accumulators' loads travel together.
template <int RT>
__device__ __forceinline__ void tmem_ld_issue(uint32_t taddr, float* v) {
  if constexpr (RT == 8)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "r"(taddr) : "memory");
  else
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]),
                   "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
                 : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_wait(float (&v)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]),
                 "+f"(v[8]), "+f"(v[9]), "+f"(v[10]), "+f"(v[11]), "+f"(v[12]), "+f"(v[13]), "+f"(v[14]), "+f"(v[15])
               :: "memory");
}
__device__ __forceinline__ void tmem_ld_wait(float (&v)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]),
                 "+f"(v[8]), "+f"(v[9]), "+f"(v[10]), "+f"(v[11]), "+f"(v[12]), "+f"(v[13]), "+f"(v[14]), "+f"(v[15]),
                 "+f"(v[16]), "+f"(v[17]), "+f"(v[18]), "+f"(v[19]), "+f"(v[20]), "+f"(v[21]), "+f"(v[22]),
                 "+f"(v[23]), "+f"(v[24]), "+f"(v[25]), "+f"(v[26]), "+f"(v[27]), "+f"(v[28]), "+f"(v[29]),
                 "+f"(v[30]), "+f"(v[31])
               :: "memory");
}
// Largest value of a warp, in every lane.
__device__ __forceinline__ float warp_max(float x) {
  float m;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(m) : "f"(x));
  return m;
}
// Sums x[0 .. N) over the warp; lane l ends with the total of element l / (32 / N).  N + 4 - log2 N shuffles
// instead of 5 N: each halving leaves a lane half as many elements.
template <int N, int O = 16>
__device__ __forceinline__ float warp_sum_scatter(const float (&x)[N], int lane) {
  if constexpr (N == 1) {
    float t = x[0];
#pragma unroll
    for (int o = O; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
  } else {
    float y[N / 2];
    const bool up = lane & O;
#pragma unroll
    for (int i = 0; i < N / 2; ++i)
      y[i] = (up ? x[i + N / 2] : x[i]) + __shfl_xor_sync(0xffffffffu, up ? x[i] : x[i + N / 2], O);
    return warp_sum_scatter<N / 2, O / 2>(y, lane);
  }
}
// Element l / (32 / N) of x for lane l.
template <int N, int O = 16>
__device__ __forceinline__ float lane_element(const float (&x)[N], int lane) {
  if constexpr (N == 1) {
    return x[0];
  } else {
    float y[N / 2];
#pragma unroll
    for (int i = 0; i < N / 2; ++i) y[i] = lane & O ? x[i + N / 2] : x[i];
    return lane_element<N / 2, O / 2>(y, lane);
  }
}

// Two fp32 values in one 64-bit register, for the packed fp32 instructions of sm_100
// (one issue slot for two results).
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t r, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(r));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// 2^f for a pair, |f| <= 0.5: degree-4 minimax polynomial (relative error 2.6e-6).
__device__ __forceinline__ uint64_t exp2_frac2(uint64_t f) {
  uint64_t p = fma2(pack2(0.009570102207f, 0.009570102207f), f, pack2(0.05591785908f, 0.05591785908f));
  p = fma2(p, f, pack2(0.2402474433f, 0.2402474433f));
  p = fma2(p, f, pack2(0.6931217909f, 0.6931217909f));
  return fma2(p, f, pack2(0.9999992847f, 0.9999992847f));
}
// p * 2^n for a pair, n in the low mantissa bits of t (the 1.5 * 2^23 rounding trick).
__device__ __forceinline__ uint64_t scale_exp2(uint64_t p, uint64_t t) {
  float t0, t1, p0, p1;
  unpack2(t, t0, t1);
  unpack2(p, p0, p1);
  return pack2(__int_as_float(__float_as_int(p0) + (__float_as_int(t0) << 23)),
               __int_as_float(__float_as_int(p1) + (__float_as_int(t1) << 23)));
}
__device__ __forceinline__ uint64_t magic2() { return pack2(12582912.0f, 12582912.0f); }
// 2^x for a pair on the FMA pipe, x in [-125, 126].
__device__ __forceinline__ uint64_t exp2_poly2(uint64_t x) {
  const uint64_t t = add2(x, magic2());
  return scale_exp2(exp2_frac2(sub2(x, sub2(t, magic2()))), t);
}
// 2^(v * c2) for a pair on the FMA pipe, the scaling folded into the range reduction.
__device__ __forceinline__ uint64_t exp2_poly_scaled2(uint64_t v, uint64_t c22) {
  const uint64_t t = fma2(v, c22, magic2());
  return scale_exp2(exp2_frac2(fma2(v, c22, sub2(magic2(), t))), t);
}
// 2^x for a pair on the special-function unit.
__device__ __forceinline__ uint64_t exp2_sfu2(uint64_t x) {
  float x0, x1;
  unpack2(x, x0, x1);
  return pack2(fast_exp2(x0), fast_exp2(x1));
}
// Which of the 16 element pairs of a chunk take the polynomial (the special-function unit gives 16
// results per clock and SM, the FMA pipe works beside it).  Fed from tensor memory alone the mixes
// reach 16.7 (pass 1, 2 pairs) to 18.3 (5) and 19.0 (pass 2, 4) to 21.2 (6) elements per clock and SM;
// inside the kernel, where every instruction beside the arithmetic takes issue slots from it, the
// shares below are the best at the power cap (128K keys, us per pass-1 / pass-2 task: 80.6 / 71.2
// with 2 and 4 pairs, 85.0 / 70.0 with 0 and 5, 81.1 / 73.4 with 3 and 6).
__host__ __device__ constexpr bool poly1(int pr) { return pr % 8 == 0; }
__host__ __device__ constexpr bool poly2(int pr) { return pr % 4 == 0; }
// Percentage of a problem's keys (its end) that pass 1 asks L2 to keep for pass 2, which walks backwards; the
// other keys make room first.  Whole prefills of 32768 keys, us, with nothing kept / with this: window 64
// 1727 / 1714, window 8 1009 / 991.
// Several row blocks of a KV group read the same keys one after the other, so among other layers none of
// them makes room first.  us with the hints / without: 16 layers of 65536 keys in two blocks 1418 / 1386, in four
// 2625 / 2545; 28 of 20001 1453 / 1428, of 5003 418 / 416; but 20 of 2048 105 / 108, and one layer of 131072
// 326 / 331.
constexpr int kL2KeepPct = 20, kL2PlainFrom = 4096;

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, rows of 128 bytes, 8-row
// groups 1024 bytes apart (the layout TMA writes with CU_TENSOR_MAP_SWIZZLE_128B).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3fffu);          // start address, 16-byte units
  d |= (uint64_t)1 << 16;                          // leading-dimension byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;                // stride between 8-row groups
  d |= (uint64_t)1 << 46;                          // descriptor version of this architecture
  d |= (uint64_t)2 << 61;                          // 128-byte swizzle
  return d;
}
// Shared-memory matrix descriptor of an unswizzled K-major operand of 16 columns (one MMA
// K-step): 8-row x 16-byte core matrices of 128 contiguous bytes, the two K halves of a row
// group 128 bytes apart, row groups 256 bytes apart.  Element (row, k) therefore sits at
// (row / 8) * 256 + (k / 8) * 128 + (row % 8) * 16 + (k % 8) * 2.
__device__ __forceinline__ uint64_t smem_desc_k16(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3fffu);
  d |= (uint64_t)(128 >> 4) << 16;                 // between the core matrices of one row group (K direction)
  d |= (uint64_t)(256 >> 4) << 32;                 // between row groups
  d |= (uint64_t)1 << 46;
  return d;
}
__device__ __forceinline__ uint32_t k16_offset(int row, int k) {
  return (uint32_t)((row >> 3) * 256 + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2);
}
// Instruction descriptor: bf16 x bf16 -> fp32, both operands K-major, tile M x N (bit 13 negates A).
__host__ __device__ constexpr uint32_t instr_desc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// ---- shared memory layout ----------------------------------------------------------------
// What a task's consumers need to know, in one piece of shared memory: parameters of the launch indexed by
// problem would be constant-memory misses on the way from one task to the next.
struct alignas(16) TcTask {
  int pass, unit, lo, hi;              // pass 0: no task left; key tiles [lo, hi)
  int n_keys, rows, row0, slot;        // score rows of the KV group from the unit's first on; that row; (problem, unit)
  float c2, v_min, inv_c2;
  int negate;
  float* cols;                         // pass 2: output of the KV group's first head
  int prob, group;
  int part, part0, n_part, n_arrive;   // pass 1: where its statistics go; the unit's partials and pass-1 tasks
  int seg, n_seg, n_pairs, pad;        // pass 1: segments [seg, seg + n_seg) of the unit's n_part over n_pairs tile pairs
};
constexpr int kTaskBytes = 96;
static_assert(sizeof(TcTask) <= kTaskBytes && sizeof(TcTask) % 16 == 0, "task slot");
template <int SH>
struct Shape {
  static constexpr bool kNarrow = SH >= kNarrow32;
  static constexpr int kRows = SH == kNarrow32 ? 32 : SH == kNarrow64 ? 64 : kRowBlock;   // score rows of a unit
  static constexpr int kW = SH == kWide16 ? 16 : SH == kWide32 ? 32 : SH == kWide64 ? 64 : SH == kWide128 ? 128 : 256;
  static constexpr int kQHalves = kNarrow ? 1 : 2;         // parts the Q block is loaded in
  static constexpr int kQBufs = kNarrow ? 2 : 1;           // Q blocks held (of wide ones two do not fit)
  static constexpr int kAcc = kNarrow ? 8 : 2;             // accumulator ring in tensor memory
  static constexpr int kFoldWarps = kNarrow ? 4 : 8;       // compute warps that store a pass-1 task's statistics
  static constexpr int kAccCols = 512 / kAcc;
};
template <int D, int SH>
struct Smem {
  static constexpr int kRows = Shape<SH>::kRows;
  static constexpr int kSub = D / 64;                      // 64-column (128-byte) sub-tiles per operand
  static constexpr int kQSub = kRows * 128;                // one sub-tile of the Q block
  static constexpr int kQBytes = kQSub * kSub;
  static constexpr int kKSub = kKeyTile * 128;             // one sub-tile of one K stage: 128 keys x 128 bytes
  static constexpr int kKBytes = kKSub * kSub;             // bytes TMA delivers per stage
  // K ring, sub-tile major: sub-tile c of stage s sits at kKOff + (c * kStages + s) * kKSub, so the
  // same sub-tile of stages s and s + 1 is one contiguous 256-key operand
  static constexpr int kKOff = kQBytes * Shape<SH>::kQBufs;
  static constexpr int kOnesOff = kKOff + kStages * kKBytes;       // extra K-step, key side: 128 x 16 bf16
  static constexpr int kExtOff = kOnesOff + kKeyTile * 32;         // extra K-step, row side: [2][kRows x 16] bf16
  static constexpr int kPartOff = kExtOff + 2 * kRows * 32;        // [2][3][kRows] partials (log-sum-exp, entropy)
  static constexpr int kTaskOff = kPartOff + 2 * 3 * kRows * 8;    // task ring
  static constexpr int kBarOff = kTaskOff + kTaskRing * kTaskBytes;
  static constexpr int kBytes = kBarOff + 512;
  static constexpr int kAlloc = kBytes + 1024;             // slack to align the base to 1024 bytes
  static_assert(kAlloc <= 227 * 1024, "shared memory of one CTA");
};

// Barrier slots (8 bytes each) inside the barrier area.
enum { kBarFull = 0, kBarEmpty = kBarFull + kStages, kBarTaskFull = kBarEmpty + kStages,
       kBarTaskEmpty = kBarTaskFull + kTaskRing, kBarQFull = kBarTaskEmpty + kTaskRing, kBarQEmpty = kBarQFull + 2,
       kBarExtFull = kBarQEmpty + 2, kBarExtEmpty = kBarExtFull + 2, kBarFold = kBarExtEmpty + 2,
       kBarPartFull = kBarFold + 4, kBarPartEmpty, kBarDrain, kBarAccFull,
       kBarAccEmpty = kBarAccFull + 8, kBarCount = kBarAccEmpty + 8 };
constexpr int kTaskConsumers = 3 + kComputeWarps;          // MMA, lse hand-over, fold, compute warps

// The four column groups (wide) or lane quarters (narrow) of a row fold into one partial, in this order; the
// thread that folds holds the own-th of them.
__device__ __forceinline__ float2 fold_row(const float2* part_s, int stride, float2 mine, int own) {
  float2 c[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) c[k] = k == own ? mine : part_s[(k < own ? k : k - 1) * stride];
  float M = -INFINITY, W = 0.f, X = 0.f;
  merge_partials(M, W, X, c);
  const float lw = __log2f(W);
  return W > 0.f ? make_float2(M + lw, lw + __fdividef(X, W)) : make_float2(-INFINITY, 0.f);
}
// Merges a unit's partials for the rows lane, lane + 32, ... of one warp, four rows (24 loads) at a time;
// done(row, -lse, entropy) with (-inf, 0) for rows that saw no key.
template <int R, typename F>
__device__ __forceinline__ void merge_unit(const float2* part, int n_part, int lane, F done) {
  constexpr int kRowsAt = R < 128 ? R / 32 : 4, kBatch = kMergeGroup;
  for (int r0 = lane; r0 < R; r0 += 32 * kRowsAt) {
    float M[kRowsAt], W[kRowsAt], X[kRowsAt];
#pragma unroll
    for (int q = 0; q < kRowsAt; ++q) { M[q] = -INFINITY; W[q] = X[q] = 0.f; }
    for (int s0 = 0; s0 < n_part; s0 += kBatch) {
      float2 pv[kRowsAt][kBatch];
#pragma unroll
      for (int b = 0; b < kBatch; ++b)
#pragma unroll
        for (int q = 0; q < kRowsAt; ++q)
          pv[q][b] = s0 + b < n_part ? __ldcg(part + (size_t)(s0 + b) * R + r0 + 32 * q) : make_float2(-INFINITY, 0.f);
#pragma unroll
      for (int q = 0; q < kRowsAt; ++q) merge_partials(M[q], W[q], X[q], pv[q]);
    }
#pragma unroll
    for (int q = 0; q < kRowsAt; ++q) {
      const float lz = __log2f(W[q]);
      done(r0 + 32 * q, W[q] > 0.f ? -(M[q] + lz) : -INFINITY, W[q] > 0.f ? kLn2 * (lz + X[q] / W[q]) : 0.f);
    }
  }
}
// Adds one chunk of 32 keys to a row's statistics, all keys visible.  False: a logit far above the
// reference overflowed (or was outside the polynomial's range) and the chunk has to be redone.
__device__ __forceinline__ bool stat_add(RowStat& r, const float (&v)[32], uint64_t c22) {
  const uint64_t nref2 = pack2(-r.ref, -r.ref);
  uint64_t Z2 = pack2(r.Z, 0.f), U2 = pack2(r.U, 0.f);
  float top = 0.f;
#pragma unroll
  for (int pr = 0; pr < 16; ++pr) {
    const uint64_t x2 = fma2(pack2(v[2 * pr], v[2 * pr + 1]), c22, nref2);
    uint64_t p2;
    if (poly1(pr)) {
      float x0, x1;
      unpack2(x2, x0, x1);
      top = fmaxf(top, fmaxf(x0, x1));
      p2 = exp2_poly2(pack2(fmaxf(x0, -125.f), fmaxf(x1, -125.f)));
    } else {
      p2 = exp2_sfu2(x2);
    }
    Z2 = add2(Z2, p2);
    U2 = fma2(p2, x2, U2);
  }
  float a, b;
  unpack2(Z2, a, b);
  r.Z = a + b;
  unpack2(U2, a, b);
  r.U = a + b;
  return r.Z < 4.0e37f && fabsf(r.U) < 3.0e38f && top < 120.f;
}
// The same for any chunk: keys beyond t_pos are masked (v[0] is key jb) and the reference first moves
// up to the chunk's maximum.
__device__ __forceinline__ void stat_add_masked(RowStat& r, const float (&v)[32], float c2, int jb, int t_pos) {
  float mx = -INFINITY;
#pragma unroll
  for (int e = 0; e < 32; ++e)
    if (jb + e <= t_pos) mx = fmaxf(mx, v[e] * c2);
  if (mx > r.ref) {
    if (r.ref != -INFINITY) {
      const float dm = r.ref - mx, f = fast_exp2(dm);
      r.U = f * fmaf(dm, r.Z, r.U);
      r.Z = f * r.Z;
    }
    r.ref = mx;
  }
  const float ref_use = (r.ref == -INFINITY) ? 0.f : r.ref;  // row has seen no key yet: all masked
#pragma unroll
  for (int e = 0; e < 32; ++e) {
    const float x = (jb + e <= t_pos) ? fmaf(v[e], c2, -ref_use) : kMasked;
    const float pr = fast_exp2(x);
    r.Z += pr;
    r.U = fmaf(pr, x, r.U);
  }
}
// sum of 2^(c2 v) over N consecutive elements; `pr0` = position of the first pair in its chunk of 16
template <int N>
__device__ __forceinline__ float sum_exp(const float* v, uint64_t c22, float v_min, int pr0 = 0) {
  uint64_t s2 = pack2(0.f, 0.f);
#pragma unroll
  for (int i = 0; i < N / 2; ++i) {
    uint64_t p2;
    if (poly2(pr0 + i))
      p2 = exp2_poly_scaled2(pack2(fmaxf(v[2 * i], v_min), fmaxf(v[2 * i + 1], v_min)), c22);
    else
      p2 = exp2_sfu2(fma2(pack2(v[2 * i], v[2 * i + 1]), c22, pack2(0.f, 0.f)));
    s2 = add2(s2, p2);
  }
  float a, b;
  unpack2(s2, a, b);
  return a + b;
}

template <int D, int SH, int MAXP, int FORM>
__global__ void __launch_bounds__(kTcThreads, 1) tc_score(const __grid_constant__ TcParams<MAXP> p) {
  using L = Smem<D, SH>;
  using S = Shape<SH>;
  constexpr bool HURRY = FORM == kHurry;
  constexpr int R = S::kRows, kQHalves = S::kQHalves;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* sm = smem_raw + (base - raw);
  const uint32_t bars = base + L::kBarOff;
  auto bar = [&](int slot) { return bars + 8u * (uint32_t)slot; };
  volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + L::kBarOff + 8 * kBarCount);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + L::kBarOff + 8 * kBarCount + 8);
  volatile int* mma_in_flight = reinterpret_cast<volatile int*>(sm + L::kBarOff + 8 * kBarCount + 16);
  volatile int* last_flag = reinterpret_cast<volatile int*>(sm + L::kBarOff + 8 * kBarCount + 24);
  auto task_slot = [&](int k) { return reinterpret_cast<TcTask*>(sm + L::kTaskOff + k * kTaskBytes); };
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) { mbar_init(bar(kBarFull + s), 1); mbar_init(bar(kBarEmpty + s), 1); }
    for (int s = 0; s < kTaskRing; ++s) { mbar_init(bar(kBarTaskFull + s), 1); mbar_init(bar(kBarTaskEmpty + s), kTaskConsumers); }
    for (int b = kBarQFull; b < kBarFold; ++b)
      mbar_init(bar(b), HURRY && b >= kBarExtFull && b < kBarExtEmpty ? R / 32 : 1);
    for (int b = 0; b < 4; ++b) mbar_init(bar(kBarFold + b), 4);
    mbar_init(bar(kBarPartFull), S::kFoldWarps);
    mbar_init(bar(kBarPartEmpty), 1);
    mbar_init(bar(kBarDrain), 1);
    for (int a = 0; a < S::kAcc; ++a) { mbar_init(bar(kBarAccFull + a), 1); mbar_init(bar(kBarAccEmpty + a), kComputeWarps); }
    *abort_flag = 0;
    *mma_in_flight = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // operands of pass 2's extra K-step: 1.0 in the first three K columns on the key side, zeros elsewhere
  for (int i = threadIdx.x; i < (kKeyTile + 2 * R) * 32 / 16; i += kTcThreads)
    reinterpret_cast<uint4*>(sm + L::kOnesOff)[i] =
        i < kKeyTile * 2 && (i & 8) == 0 ? make_uint4(0x3f803f80u, 0x00003f80u, 0u, 0u) : make_uint4(0u, 0u, 0u, 0u);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_trigger();
  pdl_wait();          // inputs, counters and statistics buffers belong to the kernels before this one until here

  // A consumer warp takes its next task: lane 0 polls (bounded), every lane reads the descriptor.
  // (With the suspending wait: helper warps sit here for a whole task and must not take issue slots.)
  auto next_task = [&](int n, TcTask& t, bool keep = false) {
    const int k = n % kTaskRing;
    int ok = 1;
    if (lane == 0)
      ok = mbar_wait_producer(bar(kBarTaskFull + k), (uint32_t)(n / kTaskRing) & 1u, abort_flag, kWaitCycles) ? 1 : 0;
    if (!__shfl_sync(0xffffffffu, ok, 0)) return false;
    asm volatile("" ::: "memory");
    t = *task_slot(k);
    asm volatile("" ::: "memory");
    if (keep) return t.pass != 0;                          // the slot is given back by task_done
    __syncwarp();
    if (lane == 0) mbar_arrive(bar(kBarTaskEmpty + k));
    return t.pass != 0;
  };
  // -lse / c2 of a row as hi + mid + lo (bf16 each: 24 bits together) into the extra K-step's operand; rows
  // that do not exist get a huge negative value so that their 2^x is 0.
  auto put_lse = [&](int buf, int r, float nlse, float inv_c2) {
    const float Lv = nlse == -INFINITY ? kMaskedAcc : nlse * inv_c2;
    const __nv_bfloat16 hi = __float2bfloat16_rn(Lv);
    const float r1 = Lv - __bfloat162float(hi);
    const __nv_bfloat16 mid = __float2bfloat16_rn(r1);
    const __nv_bfloat16 lo = __float2bfloat16_rn(r1 - __bfloat162float(mid));
    unsigned char* bx = sm + L::kExtOff + buf * (R * 32);
    *reinterpret_cast<__nv_bfloat16*>(bx + k16_offset(r, 0)) = hi;
    *reinterpret_cast<__nv_bfloat16*>(bx + k16_offset(r, 1)) = mid;
    *reinterpret_cast<__nv_bfloat16*>(bx + k16_offset(r, 2)) = lo;
  };
  auto is_row = [&](int row) { return row < p.rows_pg && (row & (p.w_pad - 1)) < p.window; };   // row of the KV group, padding excluded
  // First key tile of segment k of a pass-1 task (which holds n_seg of them).
  auto segment_lo = [](const volatile TcTask& t, int k) { return 2 * (int)((unsigned)(t.seg + k) * (unsigned)t.n_pairs / (unsigned)t.n_part); };
  // The n-th Q block: wide ones come in halves with a barrier each, narrow ones alternate between two buffers.
  auto q_bar = [](int n, int half) { return S::kQBufs == 2 ? n & 1 : half; };
  auto q_parity = [](int n) { return (uint32_t)(S::kQBufs == 2 ? n >> 1 : n) & 1u; };
  auto q_buf = [](int n) { return S::kQBufs == 2 ? (n & 1) * L::kQBytes : 0; };
  // Tiles of item `it` of a task: pass 1 ascends, pass 2 descends; half 1 may be missing at the end.
  auto tile_of = [](const TcTask& t, int it, int half) { return t.pass == 1 ? t.lo + 2 * it + half : t.hi - 1 - 2 * it - half; };
  auto present = [](const TcTask& t, int tile) { return tile >= t.lo && tile < t.hi; };
  auto items_of = [](const TcTask& t) { return (t.hi - t.lo + 1) / 2; };

  if (warp == 0) {
    // ---------------- ticket taker and TMA producer ----------------
    if (lane == 0) {
      const uint64_t pol_keep = l2_policy_evict_last(), pol_stream = l2_policy_evict_first(), pol_plain = l2_policy_evict_normal();
      int* const ticket = p.ctl + kCtlTicket;
      const int n_tickets = p.phase[p.n_phase].first;
      int tk = atomicAdd(ticket, 1), ph = 0;
      int st = 0, n_q = 0;                                 // K stages used, Q blocks loaded so far
      unsigned q_uses[2] = {0, 0};                         // copies behind each Q barrier
      unsigned real = 0;                                   // stages whose last use was a copy
      for (int n = 0;; ++n) {
        TcTask t{};
        int g = 0, rb = 0;
        if (tk < n_tickets) {
          while (tk >= p.phase[ph + 1].first) ++ph;
          t.pass = p.phase[ph].pass;
          t.prob = p.phase[ph].prob;
          t.group = p.group;
          const TcProblem& pb = p.prob[t.prob];
          const int tasks = t.pass == 1 ? pb.t1 : pb.t2;
          int i = tk - p.phase[ph].first;
          if (t.pass == 2) i = tasks - 1 - i;              // pass 2 starts with the keys pass 1 touched last
          // the unit whose share [tc_deal(W), tc_deal(W + w)) holds task i
          const int w_at = ((i + 1) * p.w_total - 1) / tasks;
          g = w_at / p.w_group;
          rb = min((w_at - g * p.w_group) / kFullWeight, p.n_rb - 1);
          const int w0 = g * p.w_group + rb * kFullWeight;
          const int i0 = tc_deal(w0, tasks, p.w_total);
          const int w_unit = rb == p.n_rb - 1 ? p.w_last : kFullWeight;
          const int n_here = tc_deal(w0 + w_unit, tasks, p.w_total) - i0;
          const int at = i - i0, n_tiles = (pb.n_keys + kKeyTile - 1) / kKeyTile;
          // the unit's segments: one partial each
          const int s0 = tc_deal(w0, pb.s1, p.w_total);
          t.n_part = tc_deal(w0 + w_unit, pb.s1, p.w_total) - s0;
          t.part0 = pb.part0 + s0;
          if (t.pass == 1) {
            t.n_arrive = n_here;
            t.seg = at * t.n_part / n_here;
            t.n_seg = (at + 1) * t.n_part / n_here - t.seg;
            t.part = t.part0 + t.seg;
            t.n_pairs = (n_tiles + 1) / 2;
            t.lo = segment_lo(t, 0);
            t.hi = segment_lo(t, t.n_seg);
            if (S::kNarrow) t.hi = min(t.hi, n_tiles);     // a wide accumulator takes a pair: the odd tile's partner is masked
          } else {
            t.n_arrive = tc_deal(w0 + w_unit, pb.t1, p.w_total) - tc_deal(w0, pb.t1, p.w_total);
            t.lo = (int)((long long)at * n_tiles / n_here);
            t.hi = (int)((long long)(at + 1) * n_tiles / n_here);
          }
          t.unit = g * p.n_rb + rb;
          t.slot = t.prob * p.n_units + t.unit;
          t.n_keys = pb.n_keys;
          t.row0 = rb * R;
          t.rows = p.rows_pg - rb * R;
          t.c2 = pb.c2; t.v_min = pb.v_min; t.inv_c2 = pb.inv_c2; t.negate = pb.negate;
          t.cols = pb.cols + (size_t)g * p.group * p.col_stride;
          tk = atomicAdd(ticket, 1);                       // travels while this task is loaded
        }
        const int k = n % kTaskRing;
        if (!mbar_wait_producer(bar(kBarTaskEmpty + k), ((uint32_t)(n / kTaskRing) & 1u) ^ 1u, abort_flag, kWaitCycles)) break;
        *task_slot(k) = t;
        mbar_arrive(bar(kBarTaskFull + k));
        if (t.pass == 0) break;
        const TcProblem& pb = p.prob[t.prob];
        const int n_tiles = (pb.n_keys + kKeyTile - 1) / kKeyTile;
        const bool plain = p.n_rb > 1 && !HURRY && pb.n_keys >= kL2PlainFrom;
        const int keep_from = t.pass == 1 && !plain ? n_tiles - (n_tiles * kL2KeepPct) / 100 : n_tiles;
        bool ok = true;
        for (int it = 0; it < items_of(t) && ok; ++it) {
          for (int half = 0; half < 2; ++half, ++st) {
            const int sg = st % kStages, tile = tile_of(t, it, half);
            ok = mbar_wait_producer(bar(kBarEmpty + sg), ((uint32_t)(st / kStages) & 1u) ^ 1u, abort_flag, kWaitCycles);
            if (!ok) break;
            if (!present(t, tile)) {
              real &= ~(1u << sg);
              mbar_arrive(bar(kBarFull + sg));
              continue;
            }
            real |= 1u << sg;
            mbar_expect_tx(bar(kBarFull + sg), L::kKBytes);
            // a tile may reach beyond the sequence's last key (into zero fill, or into the next
            // sequence of a packed batch): the causal mask discards those keys
            for (int c = 0; c < L::kSub; ++c)
              tma_load_3d_hint(base + L::kKOff + (c * kStages + sg) * L::kKSub, &p.map_k[pb.map], bar(kBarFull + sg),
                               c * 64, pb.key0 + tile * kKeyTile, g, tile >= keep_from ? pol_keep : plain ? pol_plain : pol_stream);
          }
          if (it == 0 && ok) {
            // The Q block, behind the first keys, in halves: each waits for the previous task's MMAs on it,
            // and pass 1 is done with the first half an accumulator earlier.
            const int head = pb.head0 + g * p.group + rb * (R / p.w_pad);
            for (int hq = 0; hq < kQHalves && ok; ++hq) {
              const int qb = q_bar(n_q, hq);
              ok = mbar_wait_producer(bar(kBarQEmpty + qb), q_parity(n_q) ^ 1u, abort_flag, kWaitCycles);
              if (!ok) break;
              mbar_expect_tx(bar(kBarQFull + qb), L::kQBytes / kQHalves);
              const int row = hq * (R / kQHalves);
              for (int c = 0; c < L::kSub; ++c)
                tma_load_3d_hint(base + q_buf(n_q) + c * L::kQSub + row * 128, &p.map_q[pb.map], bar(kBarQFull + qb), c * 64,
                                 row % p.w_pad, head + row / p.w_pad, pol_keep);
              ++q_uses[qb];
            }
            if (ok) ++n_q;
          }
        }
        if (!ok) break;
      }
      // every copy this thread issued must have landed before the CTA may exit (they have, unless
      // the CTA is aborting: an MMA consumed each of them)
      for (int qb = 0; qb < 2; ++qb)
        if (q_uses[qb]) mbar_drain(bar(kBarQFull + qb), (q_uses[qb] - 1u) & 1u, abort_flag);
      for (int u = max(0, st - kStages); u < st; ++u)
        if (real >> (u % kStages) & 1u) mbar_drain(bar(kBarFull + u % kStages), (uint32_t)(u / kStages) & 1u, abort_flag);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    if (lane == 0) {
      constexpr uint32_t idesc_ext = instr_desc(128, R);   // wide pass 1 has N = 256 = R as well
      const uint64_t q_desc_at = smem_desc(base), k_desc0 = smem_desc(base + L::kKOff);
      const uint64_t ones_desc = smem_desc_k16(base + L::kOnesOff), ext_desc = smem_desc_k16(base + L::kExtOff);
      int st = 0, n_q = 0, n_ext = 0, u = 0;               // K stages, tasks with items, pass-2 tasks, accumulators so far
      bool ok = true;
      auto full = [&](int s) { return mbar_wait_producer(bar(kBarFull + s % kStages), (uint32_t)(s / kStages) & 1u, abort_flag, kWaitCycles); };
      auto q_full = [&](int hq) { return mbar_wait_producer(bar(kBarQFull + q_bar(n_q, hq)), q_parity(n_q), abort_flag, kWaitCycles); };
      auto acc_free = [&]() {
        const bool r = mbar_wait_producer(bar(kBarAccEmpty + u % S::kAcc), ((uint32_t)(u / S::kAcc) & 1u) ^ 1u, abort_flag, kWaitCycles);
        tc_fence_after();
        return r;
      };
      for (int n = 0; ok; ++n) {
        const int k = n % kTaskRing;
        if (!mbar_wait_producer(bar(kBarTaskFull + k), (uint32_t)(n / kTaskRing) & 1u, abort_flag, kWaitCycles)) break;
        asm volatile("" ::: "memory");
        const TcTask t = *task_slot(k);
        asm volatile("" ::: "memory");
        mbar_arrive(bar(kBarTaskEmpty + k));
        if (t.pass == 0) break;
        const int items = items_of(t);
        if (items == 0) continue;
        const int n_half = min(R, t.rows) > 128 ? 2 : 1;
        const uint32_t idesc = idesc_ext | (t.negate ? 1u << 13 : 0u);
        const uint64_t q_desc0 = q_desc_at + (uint64_t)(q_buf(n_q) >> 4);
        for (int it = 0; it < items && ok; ++it, st += 2) {
          // descriptors differ only in the start-address field (16-byte units, no carry out of it)
          if (!S::kNarrow && t.pass == 1) {
            // accumulator = (pair, row half): A = one 128-row half of Q, B = the pair's 256 keys
            ok = full(st) && full(st + 1);
            const uint64_t kd = k_desc0 + (uint64_t)(((st % kStages) * L::kKSub) >> 4);
            for (int hf = 0; hf < n_half && ok; ++hf, ++u) {
              if (it == 0 && !(ok = q_full(hf))) break;
              if (!(ok = acc_free())) break;
#pragma unroll
              for (int kk = 0; kk < D / 16; ++kk) {
                const uint32_t qo = (kk / 4) * L::kQSub + hf * (128 * 128) + (kk % 4) * 32;
                const uint32_t ko = (kk / 4) * (kStages * L::kKSub) + (kk % 4) * 32;
                tc_mma_bf16(tmem + (u % S::kAcc) * S::kAccCols, q_desc0 + (qo >> 4), kd + (ko >> 4), idesc, kk > 0);
              }
              *mma_in_flight = 1;
              tc_commit(bar(kBarAccFull + u % S::kAcc));
              if (it == items - 1) tc_commit(bar(kBarQEmpty + hf));
            }
            if (!ok) break;
            tc_commit(bar(kBarEmpty + st % kStages));      // both K stages reusable once these MMAs have read them
            tc_commit(bar(kBarEmpty + (st + 1) % kStages));
          } else {
            // accumulator = one key tile: A = 128 keys, B = the whole Q block
            for (int half = 0; half < 2 && ok; ++half) {
              ok = full(st + half);
              if (!ok) break;
              const int sg = (st + half) % kStages;
              if (!present(t, tile_of(t, it, half))) { mbar_arrive(bar(kBarEmpty + sg)); continue; }
              if (it == 0 && half == 0)
                for (int hq = 0; hq < kQHalves && ok; ++hq) ok = q_full(hq);
              if (!ok || !(ok = acc_free())) break;
              const uint64_t kd = k_desc0 + (uint64_t)((sg * L::kKSub) >> 4);
              const uint32_t acc = tmem + (u % S::kAcc) * S::kAccCols;
#pragma unroll
              for (int kk = 0; kk < D / 16; ++kk) {
                const uint32_t ko = (kk / 4) * (kStages * L::kKSub) + (kk % 4) * 32;
                const uint32_t qo = (kk / 4) * L::kQSub + (kk % 4) * 32;
                tc_mma_bf16(acc, kd + (ko >> 4), q_desc0 + (qo >> 4), idesc, kk > 0);
              }
              *mma_in_flight = 1;
              if (t.pass == 2) {
                // one more K-step adds -lse / c2 of every row: ones (key side) x three bf16 pieces of
                // the value (row side)
                if (it == 0 && half == 0 &&
                    !(ok = mbar_wait_producer(bar(kBarExtFull + (n_ext & 1)), (uint32_t)(n_ext >> 1) & 1u, abort_flag, kWaitCycles))) break;
                tc_mma_bf16(acc, ones_desc, ext_desc + (uint64_t)((n_ext & 1) * (R * 32) >> 4), idesc_ext, 1);
              }
              tc_commit(bar(kBarEmpty + sg));              // K stage reusable once these MMAs have read it
              tc_commit(bar(kBarAccFull + u % S::kAcc));   // accumulator ready for the compute warps
              ++u;
            }
          }
        }
        if (!ok) break;
        // hand Q back (wide pass 1 did so half by half; a block of one half never used the second)
        if (S::kNarrow || t.pass == 2) {
          for (int hq = 0; hq < kQHalves; ++hq) tc_commit(bar(kBarQEmpty + q_bar(n_q, hq)));
        } else if (n_half == 1) {
          if (!(ok = q_full(1))) break;
          tc_commit(bar(kBarQEmpty + 1));
        }
        ++n_q;
        if (t.pass == 2) { tc_commit(bar(kBarExtEmpty + (n_ext & 1))); ++n_ext; }
      }
      // drain: all issued MMAs must retire before tensor memory is freed
      if (*mma_in_flight) {
        tc_commit(bar(kBarDrain));
        if (mbar_drain(bar(kBarDrain), 0, abort_flag)) *mma_in_flight = 0;
      }
    }
  } else if (warp == 2) {
    // ---------------- log-sum-exps of a pass-2 task ----------------
    int n_ext = 0;
    TcTask t;
    for (int n = 0; next_task(n, t); ++n) {
      if (HURRY || t.pass != 2 || t.lo == t.hi) continue;
      int ok = 1;
      if (lane == 0) {
        // the MMAs of the last task but one have read the operand; this unit's statistics are merged
        ok = mbar_wait_producer(bar(kBarExtEmpty + (n_ext & 1)), ((uint32_t)(n_ext >> 1) & 1u) ^ 1u, abort_flag, kWaitCycles) ? 1 : 0;
        const int* flag = p.ctl + kCtlReady + t.prob * kQueueUnits + t.unit;
        const long long t0 = clock64();
        while (ok) {
          int seen;
          asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(seen) : "l"(flag) : "memory");
          if (seen != 0) break;
          if (*abort_flag) ok = 0;
          else if ((unsigned long long)(clock64() - t0) > kWaitCycles) { *abort_flag = 1; ok = 0; }
          else __nanosleep(50);
        }
      }
      if (!__shfl_sync(0xffffffffu, ok, 0)) break;
      const size_t at0 = (size_t)t.slot * kRowBlock;
#pragma unroll
      for (int i = 0; i < R / 32; ++i) put_lse(n_ext & 1, i * 32 + lane, __ldcg(p.nlse + at0 + i * 32 + lane), t.inv_c2);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // visible to the tensor core
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(kBarExtFull + (n_ext & 1)));
      ++n_ext;
    }
  } else if (warp == 3) {
    // ---------------- row statistics of pass-1 tasks ----------------
    int n_p1 = 0;
    TcTask t;
    for (int n = 0; next_task(n, t); ++n) {
      if (HURRY || t.pass != 1) continue;
      int last = 0, ok = 1;
      if (lane == 0) {
        // the compute warps have stored the task's statistics
        ok = mbar_wait_producer(bar(kBarPartFull), (uint32_t)n_p1 & 1u, abort_flag, kWaitCycles) ? 1 : 0;
        if (ok) {
          mbar_arrive(bar(kBarPartEmpty));
          __threadfence();
          last = atomicAdd(p.ctl + kCtlArrive + t.prob * kQueueUnits + t.unit, 1) == t.n_arrive - 1;
        }
      }
      if (!__shfl_sync(0xffffffffu, ok, 0)) break;
      ++n_p1;
      if (!__shfl_sync(0xffffffffu, last, 0)) continue;
      __threadfence();
      // this task completes the unit: merge its partials into each row's log-sum-exp and entropy
      const size_t at0 = (size_t)t.slot * kRowBlock;
      merge_unit<R>(p.part + (size_t)t.part0 * R, t.n_part, lane, [&](int r, float nlse, float ent) {
        const bool row = is_row(t.row0 + r);
        __stcg(p.nlse + at0 + r, row ? nlse : -INFINITY);
        p.row_ent[at0 + r] = row ? ent : 0.f;
      });
      for (int r = R + lane; r < kRowBlock; r += 32) p.row_ent[at0 + r] = 0.f;   // rows of the block the unit does not have
      __threadfence();
      __syncwarp();
      if (lane == 0)
        asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p.ctl + kCtlReady + t.prob * kQueueUnits + t.unit), "r"(1) : "memory");
    }
  } else {
    // ---------------- compute warps ----------------
    const int quarter = warp & 3;            // tensor-memory lane quarter this warp may read
    const int sub = (warp - kHelperWarps) >> 2;   // which quarter of an accumulator's columns (or of the tiles) it takes
    const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
    float2* part_s = reinterpret_cast<float2*>(sm + L::kPartOff);
    int u = 0, n_p1 = 0, n_fold = 0, n_ext = 0;
    // Every lane polls: a barrier that has already flipped costs one test, no divergence, no broadcast
    // (with four chunks of arithmetic per accumulator and scheduler each instruction here shows).
    auto acc_full_at = [&](int u) {
      const uint32_t b = bar(kBarAccFull + u % S::kAcc), parity = (uint32_t)(u / S::kAcc) & 1u;
      bool ok = mbar_try(b, parity);
      if (!__all_sync(0xffffffffu, ok)) ok = __all_sync(0xffffffffu, mbar_wait(b, parity, abort_flag)) != 0;
      tc_fence_after();
      return ok;
    };
    auto acc_full = [&]() { return acc_full_at(u); };
    // all of this warp's loads of the accumulator have landed: one arrival per warp frees it
    auto acc_release = [&]() {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(kBarAccEmpty + u % S::kAcc));
    };
    auto acc_addr = [&]() { return tmem + lane_base + (uint32_t)((u % S::kAcc) * S::kAccCols); };
    const int ct = (int)threadIdx.x - kHelperWarps * 32;
    // Statistics of a pass-1 task: the four warps that hold parts of the same rows (wide: one lane quarter, four
    // column groups; narrow: one set of rows, four lane quarters) leave them in shared memory, meet, and one or
    // two of them fold and store them.  Two buffers: whoever writes one again has met the readers of
    // the other since.  The helper that counts the task's arrival works beside the next task.
    auto part_buf = [&](int k) { return part_s + ((n_fold & 1) * 3 + k) * R; };
    auto fold_meet = [&](int set) {
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(kBarFold + set));
      const bool ok = mbar_wait(bar(kBarFold + set), (uint32_t)n_fold & 1u, abort_flag);
      return __all_sync(0xffffffffu, ok) != 0;
    };
    auto part_stored = [&](const volatile TcTask& t) {
      __syncwarp();
      bool ok = true;
      if (lane == 0) {
        if (HURRY) {                                     // each storing warp counts for itself
          __threadfence();
          atomicAdd(p.ctl + kCtlArrive + t.prob * kQueueUnits + t.unit, 1);
        } else {                                           // the helper has seen the previous task's
          ok = mbar_wait(bar(kBarPartEmpty), ((uint32_t)n_p1 & 1u) ^ 1u, abort_flag);
          if (ok) mbar_arrive(bar(kBarPartFull));
        }
      }
      return __shfl_sync(0xffffffffu, ok, 0);
    };
    // In a hurry: R / 32 of the compute warps wait for the unit's partials and merge them, a thread per row, into
    // the extra K-step's operand (the task that holds key 0 leaves the entropies).
    auto merge_now = [&](const TcTask& t) {
      bool ok = true;
      if (lane == 0 && ct < R) {
        ok = mbar_wait(bar(kBarExtEmpty + (n_ext & 1)), ((uint32_t)(n_ext >> 1) & 1u) ^ 1u, abort_flag);
        const int* count = p.ctl + kCtlArrive + t.prob * kQueueUnits + t.unit;
        const long long t0 = clock64();
        while (ok) {
          int seen;
          asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(seen) : "l"(count) : "memory");
          if (seen >= t.n_arrive * S::kFoldWarps) break;
          if (*abort_flag) ok = false;
          else if ((unsigned long long)(clock64() - t0) > kWaitCycles) { *abort_flag = 1; ok = false; }
        }
      }
      if (!__shfl_sync(0xffffffffu, ok, 0)) return false;
      if (ct < R) {
        const float2* part = p.part + (size_t)t.part0 * R + ct;
        float M = -INFINITY, W = 0.f, X = 0.f;
        // all partials of a row in one round of loads (148 SMs, 8 units: 18 or 19), merged in the helper
        // warp's groups: the bits must not depend on who merges
        constexpr int kRounds = 4;
        for (int s0 = 0; s0 < t.n_part; s0 += kRounds * kMergeGroup) {
          float2 pv[kRounds][kMergeGroup];
#pragma unroll
          for (int b = 0; b < kRounds * kMergeGroup; ++b)
            pv[b / kMergeGroup][b % kMergeGroup] =
                s0 + b < t.n_part ? __ldcg(part + (size_t)(s0 + b) * R) : make_float2(-INFINITY, 0.f);
#pragma unroll
          for (int k = 0; k < kRounds; ++k) merge_partials(M, W, X, pv[k]);
        }
        const bool row = is_row(t.row0 + ct) && W > 0.f;
        const float lz = __log2f(W);
        put_lse(n_ext & 1, ct, row ? -(M + lz) : -INFINITY, t.inv_c2);
        if (t.lo == 0) p.row_ent[(size_t)t.slot * kRowBlock + ct] = row ? kLn2 * (lz + X / W) : 0.f;
      } else if (t.lo == 0 && ct < kRowBlock) {
        p.row_ent[(size_t)t.slot * kRowBlock + ct] = 0.f;   // rows of the block the unit does not have
      }
      if (ct < R) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // visible to the tensor core
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(kBarExtFull + (n_ext & 1)));
      }
      ++n_ext;
      return true;
    };
    TcTask t;
    bool live = true;
    // What a task needs between its segments stays in its slot, not in registers.
    auto task_done = [&](int n) {
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(kBarTaskEmpty + n % kTaskRing));
    };
    for (int n = 0; live && next_task(n, t, true); task_done(n), ++n) {
      const volatile TcTask& slot = *task_slot(n % kTaskRing);
      const int n_keys = t.n_keys;
      const float c2 = t.c2;
      const uint64_t c22 = pack2(c2, c2);
      const int last_open_key = n_keys - p.window;         // the last key every window row sees
      // a tile is "plain" when all of its keys are visible to every window row (j0 + 127 <= N - w);
      // the first (N - w + 1) / 128 tiles are
      const int first_tail_tile = (last_open_key + 1) / kKeyTile;
      if (t.pass == 1 && !S::kNarrow) {
        // An accumulator holds one 128-row half of the block x the pair's 256 keys.  This thread owns
        // row (quarter * 32 + lane) of BOTH halves (accumulators alternate between them) and the 64
        // keys [sub * 64, sub * 64 + 64) of every pair.
        float v[32] = {};
        const int row_lo = quarter * 32 + lane;
        const int rows_here = min(R, t.rows), n_half = rows_here > 128 ? 2 : 1;
        auto chunk = [&](RowStat& r, int jb, bool first, int hf) {
          // of the last pair only the chunks that hold window keys (or lie beyond the sequence) are masked
          bool careful = jb + 31 > last_open_key;
          if (first && !careful) {                          // a segment's first chunk gives the rows their reference
            float mx = v[0];
#pragma unroll
            for (int e = 1; e < 32; ++e) mx = fmaxf(mx, v[e]);
            r.ref = mx * c2;
          }
          const RowStat before = r;
          if (!careful) careful = __any_sync(0xffffffffu, !stat_add(r, v, c22));
          if (careful) {
            r = before;
            stat_add_masked(r, v, c2, jb, last_open_key + ((hf * 128 + row_lo) & (p.w_pad - 1)));
          }
        };
        // One copy of the body for both halves (instruction cache): the statistics of the two rows swap
        // places after every accumulator.  The two 32-key chunks stay unrolled, so that the second
        // load travels under the first chunk's arithmetic.
        for (int sg = 0; sg < slot.n_seg && live; ++sg) {
          const int lo = segment_lo(slot, sg), n_acc = (segment_lo(slot, sg + 1) - lo) / 2 * n_half;
          RowStat rs[2] = {{-INFINITY, 0.f, 0.f}, {-INFINITY, 0.f, 0.f}};
          for (int k = 0; k < n_acc; ++k) {
            if (!acc_full()) { live = false; break; }
            const int it = n_half == 2 ? k >> 1 : k, hf = n_half == 2 ? k & 1 : 0;
            const int jb = (lo + 2 * it) * kKeyTile + sub * 64;
            const bool warp_active = hf * 128 + quarter * 32 < rows_here;
            if (warp_active) {
              tmem_ld(acc_addr() + sub * 64, v);
              chunk(rs[0], jb, it == 0, hf);
              tmem_ld(acc_addr() + sub * 64 + 32, v);
            }
            acc_release();
            if (warp_active) chunk(rs[0], jb + 32, false, hf);
            if (n_half == 2) {
              const RowStat o = rs[0];
              rs[0] = rs[1];
              rs[1] = o;
            }
            ++u;
          }
          if (!live) break;
          // column group 0 folds the rows of the first half, column group 1 those of the second
          const float2 part0 = stat_partial(rs[0]), part1 = stat_partial(rs[1]);
          if (sub != 0) part_buf(sub - 1)[row_lo] = part0;
          if (sub != 1) part_buf(sub == 0 ? 0 : sub - 1)[128 + row_lo] = part1;
          if (!fold_meet(quarter)) { live = false; break; }
          if (sub < 2) {
            const int r = sub * 128 + row_lo;
            __stcg(&p.part[(size_t)(slot.part + sg) * R + r], fold_row(part_buf(0) + r, R, sub == 0 ? part0 : part1, sub));
          }
          ++n_fold;
        }
        if (!live || (sub < 2 && !part_stored(slot))) break;
        ++n_p1;
      } else if (t.pass == 1) {
        if constexpr (S::kNarrow) {
          // Lane = key, RT rows per thread, T tiles at a time: their waits and loads overlap (a tile by
          // itself left 500 clocks of latency bare).  A row's reference is the warp's, so that the lanes'
          // sums add up without rescaling and, scattered over the lanes, in 2 RT shuffles: with a
          // reference per lane the end of a task took 4500 clocks.  28 layers of 8192 keys, window 8:
          // 281 us before, 179 now; of 32768 keys 21.2 us a layer before, 20.8 now (the reading of K).
          constexpr int RT = R / 4, T = RT == 8 ? 4 : 1, kLanes = 32 / RT;
          float v[T * RT];
          const float masked = fmaxf(kMasked * t.inv_c2, kMaskedAcc);   // times c2: finite, and 2^x flushes to 0
          for (int sg = 0; sg < slot.n_seg && live; ++sg) {
            const int lo = segment_lo(slot, sg), hi = min((int)slot.hi, segment_lo(slot, sg + 1));
            uint64_t nref2[RT / 2], Z2[RT / 2], U2[RT / 2];  // pairs of rows: -reference, Z, U
#pragma unroll
            for (int e = 0; e < RT / 2; ++e) nref2[e] = Z2[e] = U2[e] = 0;
            for (int tile0 = lo; tile0 < hi; tile0 += T) {
              const int n_here = min(T, hi - tile0);
              for (int k = 0; k < n_here; ++k) live = live && acc_full_at(u + k);
              if (!live) break;
#pragma unroll
              for (int k = 0; k < T; ++k)
                tmem_ld_issue<RT>(tmem + lane_base + (uint32_t)(((u + min(k, n_here - 1)) % S::kAcc) * S::kAccCols) + sub * RT, v + k * RT);
              tmem_ld_wait(v);
              tc_fence_before();
              __syncwarp();
              if (lane < n_here) mbar_arrive(bar(kBarAccEmpty + (u + lane) % S::kAcc));
              u += n_here;
              const bool plain = tile0 + n_here <= first_tail_tile && n_here == T;
              if (!plain) {
#pragma unroll
                for (int k = 0; k < T; ++k) {
                  const int over = k < n_here ? (tile0 + k) * kKeyTile + quarter * 32 + lane - last_open_key : 0x7fffffff;
#pragma unroll
                  for (int e = 0; e < RT; ++e)         // rows i < over do not see this key
                    if (((sub * RT + e) & (p.w_pad - 1)) < over) v[k * RT + e] = masked;
                }
              }
              // largest logit of rows 2 e and 2 e + 1 over the warp's keys of these tiles
              auto row_max = [&](int e, float& m0, float& m1) {
                m0 = v[2 * e];
                m1 = v[2 * e + 1];
#pragma unroll
                for (int k = 1; k < T; ++k) {
                  m0 = fmaxf(m0, v[k * RT + 2 * e]);
                  m1 = fmaxf(m1, v[k * RT + 2 * e + 1]);
                }
                m0 = warp_max(m0) * c2;
                m1 = warp_max(m1) * c2;
              };
              if (tile0 == lo) {                           // the references: where a task starts, unless masked
#pragma unroll
                for (int e = 0; e < RT / 2; ++e) {
                  float m0, m1;
                  row_max(e, m0, m1);
                  nref2[e] = pack2(m0 > 0.5f * masked * c2 ? -m0 : 0.f, m1 > 0.5f * masked * c2 ? -m1 : 0.f);
                }
              }
              float top = -INFINITY;
#pragma unroll
              for (int i = 0; i < T * RT / 2; ++i) {
                const uint64_t x2 = fma2(pack2(v[2 * i], v[2 * i + 1]), c22, nref2[i % (RT / 2)]);
                float x0, x1;
                unpack2(x2, x0, x1);
                top = fmaxf(top, fmaxf(x0, x1));
              }
              if (__any_sync(0xffffffffu, top > 60.f)) {     // far above the references: they move up
#pragma unroll
                for (int e = 0; e < RT / 2; ++e) {
                  float m[2], r[2], z[2], w[2];
                  row_max(e, m[0], m[1]);
                  unpack2(nref2[e], r[0], r[1]);
                  unpack2(Z2[e], z[0], z[1]);
                  unpack2(U2[e], w[0], w[1]);
#pragma unroll
                  for (int h = 0; h < 2; ++h)
                    if (m[h] > -r[h]) {
                      const float dm = -r[h] - m[h], f = fast_exp2(dm);
                      w[h] = f * fmaf(dm, z[h], w[h]);
                      z[h] *= f;
                      r[h] = -m[h];
                    }
                  nref2[e] = pack2(r[0], r[1]);
                  Z2[e] = pack2(z[0], z[1]);
                  U2[e] = pack2(w[0], w[1]);
                }
              }
#pragma unroll
              for (int i = 0; i < T * RT / 2; ++i) {
                const uint64_t x2 = fma2(pack2(v[2 * i], v[2 * i + 1]), c22, nref2[i % (RT / 2)]), p2 = exp2_sfu2(x2);
                Z2[i % (RT / 2)] = add2(Z2[i % (RT / 2)], p2);
                U2[i % (RT / 2)] = fma2(p2, x2, U2[i % (RT / 2)]);
              }
            }
            if (!live) break;
            float ref[RT], Z[RT], U[RT];
#pragma unroll
            for (int e = 0; e < RT / 2; ++e) {
              unpack2(nref2[e], ref[2 * e], ref[2 * e + 1]);
              unpack2(Z2[e], Z[2 * e], Z[2 * e + 1]);
              unpack2(U2[e], U[2 * e], U[2 * e + 1]);
            }
            const float ref_l = -lane_element(ref, lane), Z_l = warp_sum_scatter(Z, lane), U_l = warp_sum_scatter(U, lane);
            const float2 part = stat_partial(RowStat{Z_l > 0.f ? ref_l : -INFINITY, Z_l, U_l});
            const int r = sub * RT + lane / kLanes;
            if (quarter != 0 && lane % kLanes == 0) part_buf(quarter - 1)[r] = part;
            if (!fold_meet(sub)) { live = false; break; }
            if (quarter == 0 && lane % kLanes == 0)
              __stcg(&p.part[(size_t)(slot.part + sg) * R + r], fold_row(part_buf(0) + r, R, part, 0));
            ++n_fold;
          }
          if (!live || (quarter == 0 && !part_stored(slot))) break;
          ++n_p1;
        }
      } else {
        // Pass 2: this thread owns key (tile * 128 + quarter * 32 + lane); x = c2 * accumulator.
        if (HURRY && t.hi > t.lo && !merge_now(t)) break;
        const float v_min = t.v_min, inv_w = 1.0f / (float)p.window;
        // Columns (rows of the block) this warp sums: a quarter of them on every tile, or, where a
        // head spans more, the head's rows on every second or fourth tile, so that a head's column
        // sum never spans two warps.  Narrow blocks: all rows on every fourth tile.
        constexpr int kW = S::kW;
        constexpr bool kEighths = S::kNarrow || kW == 16;   // heads of 8 .. 64 rows, summed eight rows at a time
        constexpr int kCols = S::kNarrow ? R : kW <= 64 ? 64 : kW;
        const int turn = S::kNarrow || kW == 256 ? 3 : kW == 128 ? 1 : 0;
        const int col0 = S::kNarrow || kW == 256 ? 0 : kW == 128 ? (sub & 1) * 128 : sub * 64;
        const int my_turn = kW == 128 && !S::kNarrow ? sub >> 1 : sub;
        const bool warp_active = col0 < t.rows;
        const int h0 = (t.row0 + col0) >> p.w_shift, h_end = t.group;   // heads within the KV group
        constexpr int kCopies = FORM == kBrief ? 1 : 2;
        for (int i = 0; i < t.hi - t.lo; ++i) {
          if (!acc_full()) { live = false; break; }
          const int tile = t.hi - 1 - i;
          const int j = tile * kKeyTile + quarter * 32 + lane;
          const bool plain = tile < first_tail_tile;
          const int i_min = j - last_open_key;              // window rows i < i_min do not see key j
          const bool mine = warp_active && (u & turn) == (my_turn & turn);
          const uint32_t taddr = acc_addr() + col0;
          float tot = 0.f;
          int head = h0;
#pragma unroll kCopies
          for (int c = 0; c < kCols; c += 32) {
            float v[32] = {};
            if (mine) tmem_ld(taddr + c, v);
            if (c == kCols - 32) acc_release();             // every load of the tile has landed
            if (!mine) continue;
            if (!plain) {
              // a tile that holds window keys: row e of the chunk is window row (col0 + c + e) % w_pad
#pragma unroll
              for (int e = 0; e < 32; ++e)
                if (((col0 + c + e) & (p.w_pad - 1)) < i_min) v[e] = kMaskedAcc;
            }
            auto finish_head = [&]() {
              if (head < h_end && j < n_keys) t.cols[(size_t)head * p.col_stride + j] = tot * inv_w;
              ++head;
              tot = 0.f;
            };
            if constexpr (kEighths) {
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
  }

  // ---------------- teardown ----------------
  tc_fence_before();
  __syncthreads();
  if (*abort_flag && threadIdx.x == 0) atomicCAS(p.status, 0, (int)STRUCTKV_ERR_TIMEOUT);
  // tensor memory is freed only when no MMA of this CTA can still write to it
  if (warp == 1 && !*mma_in_flight) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
  // the last CTA leaves the counters as it found them: zero
  if (threadIdx.x == 0) *last_flag = atomicAdd(p.ctl + kCtlExit, 1) == (int)gridDim.x - 1;
  __syncthreads();
  if (*last_flag) {
    for (int i = threadIdx.x; i < p.n_prob * kQueueUnits; i += kTcThreads)
      if ((i & (kQueueUnits - 1)) < p.n_units) p.ctl[kCtlArrive + i] = p.ctl[kCtlReady + i] = 0;
    if (threadIdx.x == 0) p.ctl[kCtlTicket] = p.ctl[kCtlExit] = 0;
  }
}

template <int D, int SH, int MAXP>
cudaError_t tc_launch(const TcParams<MAXP>& p, int grid, int device, cudaStream_t st) {
  // (one problem is in a hurry)
  const auto kern = MAXP == 1 || p.form == kHurry ? tc_score<D, SH, MAXP, kHurry>
                    : p.form == kBrief            ? tc_score<D, SH, MAXP, MAXP == 1 ? kHurry : kBrief>
                                                  : tc_score<D, SH, MAXP, MAXP == 1 ? kHurry : kAmong>;
  static std::atomic<unsigned long long> ready_for[3];    // devices whose shared-memory limit has been raised
  std::atomic<unsigned long long>& ready = ready_for[p.form];
  const unsigned long long bit = 1ull << (device & 63);
  if (!(ready.load(std::memory_order_acquire) & bit)) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Smem<D, SH>::kAlloc);
    if (e != cudaSuccess) return e;
    ready.fetch_or(bit, std::memory_order_release);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kTcThreads);
  cfg.dynamicSmemBytes = Smem<D, SH>::kAlloc;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  void* args[1] = {const_cast<TcParams<MAXP>*>(&p)};        // no copies of a parameter block of kilobytes
  return cudaLaunchKernelExC(&cfg, (const void*)kern, args);
}
#endif  // __CUDACC__

// A 3-D tensor map of bf16 rows of head_dim elements, 128-byte swizzle: extents d1 x d2 of strides s1, s2 (bytes),
// boxes of b1 x b2 rows.
bool tc_encode3(const Ctx& ctx, CUtensorMap* m, const void* base, cuuint64_t d1, cuuint64_t d2, cuuint64_t s1,
                cuuint64_t s2, cuuint32_t b1, cuuint32_t b2);

// One translation unit per head dimension and parameter size instantiates the kernels.
cudaError_t tc_launch_64(int shape, const TcParams<1>& p, int grid, int device, cudaStream_t st);
cudaError_t tc_launch_64(int shape, const TcParams<kMaxBatch>& p, int grid, int device, cudaStream_t st);
cudaError_t tc_launch_128(int shape, const TcParams<1>& p, int grid, int device, cudaStream_t st);
cudaError_t tc_launch_128(int shape, const TcParams<kMaxBatch>& p, int grid, int device, cudaStream_t st);

}  // namespace skv
