// Internal declarations shared by the translation units of libstructkv (not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "structkv.h"

namespace skv {

constexpr int kKeyTile = 128;        // keys per tile in every scorer
constexpr int kMaxSms = 160;          // SMs a scorer launch uses at most (bounds its pass-1 tasks)
constexpr int kSimtParts = 64;        // key segments per score row of the CUDA-core scorer
constexpr int kRowBlock = 256;       // score rows (head, window row) per tensor-core row block
constexpr int kMaxBatch = 32;        // sequences one batched scoring call may hold
constexpr int kMaxStatLayers = 128;   // layers one batched head-statistics call may cover
constexpr int kMaxGatherLayers = 128; // layers one multi-layer gather may cover (their pointers are a kernel argument)
constexpr int kQueueUnits = 256;      // (KV group, row block) units of one problem the tensor-core scorer can hold
constexpr int kCtlInts = 64 + 2 * kMaxBatch * kQueueUnits;   // its control block: tickets, arrivals, ready flags
constexpr int kXchSlots = 17;          // units of an exchange ring of the resident scorer's teams
constexpr int kResRows = 32;           // score rows of one of its units, at most
constexpr int kDirectTeam = 20;        // CTAs of a team that merges partials directly (score_res.cuh)
constexpr int kRefSlots = 32;          // units of a ring of common references, which larger teams have
// Tagged 64-bit words: two for every row and CTA of the teams' rings (the CUDA-core scorer needs fewer), then the rings of
// references.
constexpr int kXchPairs = kMaxSms * kXchSlots * kResRows;
constexpr int kXchWords = 2 * kXchPairs + kMaxSms / (kDirectTeam + 1) * kRefSlots * kResRows;
constexpr int kCtlExit = 1, kCtlTag = 2;   // in the control block: CTAs that are done; last tag of the exchange words
constexpr unsigned long long kWaitCycles = 1000000000ull;   // bound of a device wait, about 0.5 s at the maximum SM clock
constexpr int kMergeGroup = 6;         // partials of a row merged together
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

// Device status word values are structkv_status codes; 0 = nothing recorded.
struct Workspace {
  int* status;          // [64] ints, word 0 is the status
  int* ctl;             // [kCtlInts], follows the status block; zero between scorer launches (a launch leaves it zero)
  float2* row_part;     // partial softmax statistics of score rows: CUDA cores [kSimtParts][rows_pad], tensor cores
                        // [pass-1 task][kRowBlock]
  float* row_lse2;      // [rows_pad] negated log2-domain log-sum-exp of each score row (tensor cores)
  float* row_ent;       // [rows_pad] entropy of each score row (nats), 0 where there is no row
  float* cols;          // [H][n_pad] pooled per-head attention when the caller passes none
  float* head_part;     // [kMaxStatLayers][H][4] per-(layer, head) {sum of squared deviations from 1/n, top-k mass}
  int* stat_ctr;        // [kMaxStatLayers] and, behind it, chunk_ctr [n_pad / kKeyTile]: zero between launches
  int* chunk_ctr;
  size_t ctr_bytes;     // from `status` to here: counters
  unsigned long long* xch;   // [kXchWords] tagged words the CTAs of the one-pass scorers exchange; zero at first
  size_t zero_bytes;    // from `status` on: what starts from zero
  size_t bytes;
};

struct Ctx {
  structkv_config cfg;
  Workspace ws;
  int device;
  int sm_count;
  int rows;             // H * w
  int w_pad;            // rows a head occupies in a scorer's row blocks: w up to a power of two, at least 8
  int rows_pad;         // rows per KV group (heads at w_pad rows) padded to kRowBlock, times H_kv
  int n_pad;            // max_seq rounded up to kKeyTile
  int short_ctas = 0;   // CTAs of score_short.cuh's launches, at most; 0: one per task
  bool old_words;       // the exchange words hold anything (a call's own context): who uses them clears them first
  void* tc;             // tensor-core scorer state (tensor-map encoder), owned by score_tc.cu
  struct HostSlot* slot = nullptr;   // where the device leaves the pivot for the host (api.cu), taken at first use
};

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Carves the workspace; with base == nullptr only the size is computed.
Workspace carve_workspace(const structkv_config& cfg, void* base);

// What a launch that uses the exchange words does first.
inline cudaError_t clean_words(const Ctx& ctx, cudaStream_t st) {
  return ctx.old_words ? cudaMemsetAsync(ctx.ws.xch, 0, kXchWords * sizeof(unsigned long long), st) : cudaSuccess;
}

// ---- launchers (each returns cudaGetLastError() of its launches) -------------------------
// Both scorer passes over `n` problems: layers of one shape, or (tensor cores only) the sequences of a
// packed batch.
struct ScoreCall {
  int n;                          // layers, or sequences
  const void* const* q;           // layers: [n]; batch: one tensor [n, H, w, d]
  const void* const* k;           // layers: [n]; batch: one packed tensor
  const float* scale;             // layers: [n]; batch: one
  const int* cu_seqlens;          // batch: host, [n + 1]; NULL for layers
  long long k_stride_head, k_stride_token;   // elements
  int n_keys;                     // keys of a layer
  float* cols;                    // layer l at cols + l * cols_layer_stride; sequence b at column cu_seqlens[b]
  long long cols_layer_stride, col_stride;
  float2* part;                   // tensor cores: tc_part_tasks(...) * kRowBlock entries; CUDA cores: simt_part_entries(...)
  float* nlse;                    // tensor cores: [min(n, kMaxBatch)][rows_pad]
  float* row_ent;                 // [n][rows_pad]
};
// CUDA cores: fp32 storage, and what the tensor-core scorer does not take.
size_t simt_part_entries(const structkv_config& cfg, int n);
cudaError_t launch_score_simt(const Ctx& ctx, const ScoreCall& a, cudaStream_t st);
// Tensor cores (tcgen05): bf16 storage; one launch per kMaxBatch layers.
bool tc_supported(const Ctx& ctx, long long k_stride_head, long long k_stride_token);
int tc_window_pad(int window);
// pass-1 tasks (partial statistics of kRowBlock rows) a launch over n problems needs room for
size_t tc_part_tasks(const structkv_config& cfg, int n, bool batch);
structkv_status tc_create(Ctx& ctx);
void tc_destroy(Ctx& ctx);
cudaError_t launch_score_tc(const Ctx& ctx, const ScoreCall& a, cudaStream_t st);
// The form of it for sequences whose probabilities fit the chip's tensor memory (score_res.cu).
bool res_supported(const Ctx& ctx, const ScoreCall& a);
cudaError_t launch_score_res(const Ctx& ctx, const ScoreCall& a, int first, int n, cudaStream_t st);

// One thread waits (bounded by limit_cycles) on a barrier nobody arrives on, then records
// STRUCTKV_ERR_TIMEOUT in *status.
cudaError_t launch_wait_probe(unsigned long long limit_cycles, int* status, cudaStream_t st);

// After the scorer passes of n_layers layers: S^(l)_j = sum_h cols[l][h][j] (rows s_stride apart), C <-
// lambda C + S^(l) carried from layer to layer if c_inout, metrics[l][0] from row_ent[l][rows_pad] (Eq. 4) and
// metrics[l][1..2] from the pooled per-head attention (Eq. 5-6) or NaN.
cudaError_t launch_finish_layers(const Ctx& ctx, const float* cols, long long layer_stride, long long col_stride, int n,
                                 int n_layers, float lambda, float* s_out, long long s_stride, float* c_inout,
                                 const float* row_ent, bool with_head_stats, float* metrics, cudaStream_t st,
                                 bool c_from_zero = false);
// The same for the sequences of a packed batch (sequence b at column cu_seqlens[b] of cols, s_out and c_inout).
cudaError_t launch_finish_packed(const Ctx& ctx, const float* cols, long long col_stride, const int* cu_seqlens, int batch,
                                 float lambda, float* s_out, float* c_inout, const float* row_ent, float* head_part,
                                 bool with_head_stats, float* metrics, cudaStream_t st);

// Eq. 5-6 for n_layers layers at once from their pooled per-head attention: writes metrics[l][1..2].
cudaError_t launch_head_stats_batch(const Ctx& ctx, const float* cols, long long layer_stride, long long col_stride,
                                    int n_layers, int n, float* metrics, cudaStream_t st);

cudaError_t launch_accumulate(const float* s_hist, long long row_stride, int pivot, int n,
                              float lambda, float* c_out, cudaStream_t st);

// Eq. 7-9 on the device (n_layers <= kMaxStatLayers), then launch_accumulate at that pivot.  `host` (mapped memory)
// receives the pivot in word 0 and T_l [n_layers] from word 1 on, each below the tag in the upper half, in any order.
cudaError_t launch_accumulate_at_pivot(const float* s_hist, long long row_stride, int n_layers, int n, float lambda,
                                       const float* metrics, const float* weights, int l_limit, float* c_out,
                                       unsigned long long* host, unsigned tag, cudaStream_t st);

// One more vector of a selection, with its own budget and output.
struct SelectExtra { const float* scores; int budget; int* idx_out; };
cudaError_t launch_select(const float* scores, long long row_stride, int batch, int n, int budget,
                          int window, int* idx_out, cudaStream_t st, const SelectExtra* extra = nullptr);
// The same for packed sequences of different lengths and budgets; rows are padded with -1.
cudaError_t launch_select_packed(const float* scores, const int* cu_seqlens, const int* budgets, int batch, int window,
                                 int* idx_out, long long idx_stride, cudaStream_t st);

cudaError_t launch_block_scores(const float* scores, long long row_stride, int batch, int n, int block_size,
                                float* out, cudaStream_t st);
cudaError_t launch_mass_recovery(const float* scores, long long row_stride, int batch, int n, const int* idx,
                                 int n_idx, float* out, int* status, cudaStream_t st);

// 4-byte rows (aligned) of a second source, gathered by the same list as a compaction of one slab.
struct CompactWords { const void* src; long long row_stride; void* dst; };
cudaError_t launch_compact(const void* src, long long slab_stride, long long row_stride,
                           int row_bytes, int n_slabs, int n_rows_src, const int* idx,
                           long long idx_slab_stride, int n_idx, void* dst, int* status, int sm_count,
                           cudaStream_t st, const CompactWords* words = nullptr);
cudaError_t launch_compact_layers(const void* const* srcs, int n_layers, long long slab_stride, long long row_stride,
                                  int row_bytes, int n_slabs, int n_rows_src, const int* idx,
                                  long long idx_layer_stride, int n_idx, void* dst, long long dst_layer_stride,
                                  int* status, int sm_count, cudaStream_t st);
// Rows of n_slabs slabs by one list.
struct CompactRows {
  const void* src;
  long long slab_stride, row_stride;
  int row_bytes, n_slabs, n_rows_src;
  const int* idx;
  int n_idx;
  void* dst;
};
// A gather of several layers (sources srcs), one of a single slab and the words that go with it in one launch.  False: not in
// that form (16-byte units, one launch each).
bool launch_compact_prefill(const CompactRows& kv, const void* const* srcs, int n_layers, long long idx_layer_stride,
                            long long dst_layer_stride, const CompactRows& other, const CompactWords& words, int* status, int sm_count,
                            cudaStream_t st, cudaError_t* e);
cudaError_t launch_group_saliency(const float* head_cols, long long col_stride, int n_heads, int group, int n,
                                  float* out, cudaStream_t st);

// Programmatic dependent launch: a kernel launched with launch_pdl() may begin (block scheduling,
// its own set-up) while the kernel before it in the stream is still draining.  pdl_trigger() lets
// the next kernel begin; pdl_wait() returns once the previous kernel has completed and its
// writes are visible, and must precede the first access to anything that kernel wrote or read.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}
// The same with clusters of CL CTAs.
template <int CL, typename... KArgs, typename... Args>
inline cudaError_t launch_cluster(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                  Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
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

// The same for a kernel of one argument whose blocks wait for one another: all of them run at once, or the launch is refused.
template <typename Arg>
inline cudaError_t launch_cooperative(void (*kernel)(Arg), dim3 grid, dim3 block, size_t smem, cudaStream_t st, const Arg& arg) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeCooperative;
  attr[1].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  void* args[1] = {const_cast<Arg*>(&arg)};              // no copies of a parameter block of kilobytes
  return cudaLaunchKernelExC(&cfg, (const void*)kernel, args);
}

// Adds one to a word of shared memory if `counts`; predicated, for a branch around it takes three times the instructions.
__device__ __forceinline__ void count_if(bool counts, unsigned* word) {
  asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %1, 0;\n@p red.shared.add.u32 [%0], 1;\n}"
               ::"r"((unsigned)__cvta_generic_to_shared(word)), "r"((unsigned)counts) : "memory");
}

__device__ __forceinline__ void add_to(float4& s, const float4& v) { s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w; }
__device__ __forceinline__ void add_to(float& s, float v) { s += v; }

// 2^x on the special-function unit (relative error about 2^-22; denormal results flush to 0).
__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// One row's softmax statistics over some keys: Z = sum 2^(x - ref), U = sum 2^(x - ref) (x - ref).
struct RowStat { float ref, Z, U; };

// A row's partial as it is stored: (l, h), its log-sum-exp l = ref + log2 Z and the entropy of the
// softmax over its keys alone, h = log2 Z - U / Z (both in bits); (-inf, 0) where it saw no key of the
// row.  Over a row's partials, lse = log2 sum 2^l and with w = 2^(l - lse) the row's entropy is
// sum w (h + lse - l)  (Eq. 4, one row).  The compute warps take the logarithm and the division, and
// loads of four rows are in flight together: merging is one warp's work beside sixteen busy ones,
// and pass 2 waits for it (18 partials of 256 rows: 35 us with one row and one logarithm at a time).
__device__ __forceinline__ float2 stat_partial(const RowStat& r) {
  const float lz = __log2f(r.Z);
  return r.Z > 0.f ? make_float2(r.ref + lz, lz - __fdividef(r.U, r.Z)) : make_float2(-INFINITY, 0.f);
}
// Adds partials to (M, W, X): lse so far = M + log2 W, X = sum 2^(l - M) (h - l + M).
template <int N>
__device__ __forceinline__ void merge_partials(float& M, float& W, float& X, const float2 (&pv)[N]) {
  float top = M;
#pragma unroll
  for (int b = 0; b < N; ++b) top = fmaxf(top, pv[b].x);
  if (top == -INFINITY) return;
  const float d = M == -INFINITY ? 0.f : M - top, f = fast_exp2(d);
  X = f * fmaf(-d, W, X);
  W *= f;
  M = top;
#pragma unroll
  for (int b = 0; b < N; ++b) {
    const float e = pv[b].x == -INFINITY ? -200.f : pv[b].x - top, w = fast_exp2(e);
    W += w;
    X = fmaf(w, pv[b].y - e, X);
  }
}
}  // namespace skv
