// CUDA-core scorer: window logits, row softmax statistics (pass 1) and pooled per-head attention columns
// (pass 2), all layers of a call in one launch per pass, or, where all blocks of a call run at once, in one
// launch that multiplies once.  Serves fp32 storage and what the tensor-core scorer does not take.  Everything is
// fp32 arithmetic in the log2 domain.
//
// Score rows are numbered as in the tensor-core scorer: row (h, i) of KV group g = h / G lives at
// g * rows_pg_pad + (h % G) * w_pad + i.  A block multiplies 128 rows with 64 keys, 8 x 4 per thread,
// both operands in shared memory with the head dimension outermost: 32 multiply-adds, two an instruction, for three
// 16-byte loads.  Bound by the FMA pipe on long sequences and by latency on short ones (8 heads,
// window 32, head dim 64, 2048 keys: a layer took 15 + 21 + 18 us with one dot product per lane, a
// pass that merged the partials and one key per thread; four layers now take 25 us with their sums).
// Instructions count on both: divisions by the rows a head occupies (a power of two), one multiply-add at a time, 96
// shuffles and eight logarithms a thread to fold eight rows over 16 threads took 4 layers of 5000 keys 76.8 us, now 69.0;
// 8 layers of 4096 92.5, now 84.1; 2 of 700 20.7, now 18.2; the whole prefill of 4 layers of 2048 keys 37.6, now 34.0.
#include <algorithm>
#include <atomic>

#include "tagged.cuh"

namespace skv {
namespace {

constexpr int kSmRows = 128, kSmKeys = 64, kSmThreads = 256;
constexpr int kSmLayers = 32;              // layers per launch (their pointers are a kernel argument)

struct SimtArgs {
  const void *q[kSmLayers], *k[kSmLayers];
  float c2[kSmLayers];
  long long sh, st;
  int N, w, w_pad, w_shift, group, rows_pg,   // w_pad = 1 << w_shift: rows a head occupies
      rows_pg_pad, rows_pad, n_rt, parts, n_keys_tiles;
  float2* part;                            // [layer][parts][rows_pad]
  float* row_ent;                          // [layer][rows_pad]
  float* cols;
  long long cols_layer_stride, col_stride;
  unsigned long long* xch;                 // one launch: tagged words
  int *ctl, *status;
};

__device__ __forceinline__ float4 load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16),
                     __uint_as_float(u.y & 0xffff0000u));
}

template <int D>
struct SimtShared {
  float q[D][kSmRows + 4];                 // [column][row]
  float k[D][kSmKeys + 4];
  union {
    float lse[kSmRows];                    // pass 2: -log2-sum-exp of the tile's rows
    float2 half[kSmRows];
  };
  float col[kSmRows / 8][kSmKeys];         // pass 2: sums over eight rows
};

// Stages 128 score rows (tile rt of group g) with the head dimension outermost; padding is zero.
template <typename T, int D>
__device__ __forceinline__ void stage_rows(const SimtArgs& a, const T* q, int g, int rt, float (*dst)[kSmRows + 4]) {
  for (int x = threadIdx.x; x < kSmRows * (D / 4); x += kSmThreads) {
    const int r = x % kSmRows, c = x / kSmRows * 4, row = rt * kSmRows + r, i = row & (a.w_pad - 1);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (row < a.rows_pg && i < a.w) v = load4(q + ((size_t)(g * a.group + (row >> a.w_shift)) * a.w + i) * D + c);
    dst[c][r] = v.x; dst[c + 1][r] = v.y; dst[c + 2][r] = v.z; dst[c + 3][r] = v.w;
  }
}
template <typename T, int D>
__device__ __forceinline__ void stage_keys(const SimtArgs& a, const T* k, int j0, float (*dst)[kSmKeys + 4]) {
  for (int x = threadIdx.x; x < kSmKeys * (D / 4); x += kSmThreads) {
    const int r = x % kSmKeys, c = x / kSmKeys * 4;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (j0 + r < a.N) v = load4(k + (size_t)(j0 + r) * a.st + c);
    dst[c][r] = v.x; dst[c + 1][r] = v.y; dst[c + 2][r] = v.z; dst[c + 3][r] = v.w;
  }
}
// acc[r][c] = q(row tr * 8 + r) . k(key tc * 4 + c)
template <int D>
__device__ __forceinline__ void multiply(const SimtShared<D>& s, int tr, int tc, float (&acc)[8][4]) {
  unsigned long long sum[8][2] = {};                       // pairs of keys
  auto both = [](float v) { unsigned long long x; asm("mov.b64 %0, {%1, %1};" : "=l"(x) : "f"(v)); return x; };
#pragma unroll 4
  for (int d = 0; d < D; ++d) {
    const float4 q0 = *reinterpret_cast<const float4*>(&s.q[d][tr * 8]), q1 = *reinterpret_cast<const float4*>(&s.q[d][tr * 8 + 4]);
    const ulonglong2 kv = *reinterpret_cast<const ulonglong2*>(&s.k[d][tc * 4]);
    const float qr[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const unsigned long long qq = both(qr[r]);
      asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(sum[r][0]) : "l"(qq), "l"(kv.x));
      asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(sum[r][1]) : "l"(qq), "l"(kv.y));
    }
  }
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[r][0]), "=f"(acc[r][1]) : "l"(sum[r][0]));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[r][2]), "=f"(acc[r][3]) : "l"(sum[r][1]));
  }
}

// Adds a tile's logits to the statistics of the thread's eight rows.
__device__ __forceinline__ void add_tile(const SimtArgs& a, const float (&acc)[8][4], int rt, int j0, float c2, RowStat (&st)[8]) {
  const int tr = threadIdx.x >> 4, tc = threadIdx.x & 15;
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int t_pos = a.N - a.w + ((rt * kSmRows + tr * 8 + r) & (a.w_pad - 1));      // the row's position: it sees keys <= t_pos
    float x[4], mx = -INFINITY;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      x[c] = j0 + tc * 4 + c <= t_pos && j0 + tc * 4 + c < a.N ? acc[r][c] * c2 : -INFINITY;
      mx = fmaxf(mx, x[c]);
    }
    if (mx > st[r].ref) {
      if (st[r].ref != -INFINITY) {
        const float dm = st[r].ref - mx, f = fast_exp2(dm);
        st[r].U = f * fmaf(dm, st[r].Z, st[r].U);
        st[r].Z *= f;
      }
      st[r].ref = mx;
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (x[c] != -INFINITY) {
        const float dx = x[c] - st[r].ref, pe = fast_exp2(dx);
        st[r].Z += pe;
        st[r].U = fmaf(pe, dx, st[r].U);
      }
  }
}
// op over the 16 threads of each of eight rows; thread t of the 16 ends with row t / 2.  Each halving leaves a thread half as
// many rows (8 shuffles instead of 32), in the order of a butterfly.
template <typename F>
__device__ __forceinline__ float over_row(const float (&x)[8], F op) {
  const bool u8 = threadIdx.x & 8, u4 = threadIdx.x & 4, u2 = threadIdx.x & 2;
  float y[4], z[2];
#pragma unroll
  for (int i = 0; i < 4; ++i) y[i] = op(u8 ? x[i + 4] : x[i], __shfl_xor_sync(0xffffffffu, u8 ? x[i] : x[i + 4], 8));
#pragma unroll
  for (int i = 0; i < 2; ++i) z[i] = op(u4 ? y[i + 2] : y[i], __shfl_xor_sync(0xffffffffu, u4 ? y[i] : y[i + 2], 4));
  const float v = op(u2 ? z[1] : z[0], __shfl_xor_sync(0xffffffffu, u2 ? z[0] : z[1], 2));
  return op(v, __shfl_xor_sync(0xffffffffu, v, 1));
}
// The 16 threads of a row fold into one partial; done(r, partial) in one of them, row r of the thread's eight.
template <typename F>
__device__ __forceinline__ void fold_rows(const RowStat (&st)[8], F done) {
  auto sum = [](float a, float b) { return a + b; };
  float x[8], u[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) x[r] = st[r].ref;
  const float M = over_row(x, [](float a, float b) { return fmaxf(a, b); });
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const float Mr = __shfl_sync(0xffffffffu, M, (threadIdx.x & 16) | 2 * r);
    const float dm = st[r].ref == -INFINITY ? 0.f : st[r].ref - Mr, f = fast_exp2(dm);
    x[r] = f * st[r].Z;
    u[r] = f * fmaf(dm, st[r].Z, st[r].U);
  }
  const float Z = over_row(x, sum), U = over_row(u, sum);
  if ((threadIdx.x & 1) == 0) done((int)(threadIdx.x & 15) >> 1, stat_partial(RowStat{M, Z, U}));
}
// Merges the partials [lo, hi) of a row, get(p): in batches of eight.
template <typename F>
__device__ __forceinline__ void merge_range(int lo, int hi, float& M, float& W, float& X, F get) {
  constexpr int kBatch = 8;
  for (int p0 = lo; p0 < hi; p0 += kBatch) {
    float2 pv[kBatch];
#pragma unroll
    for (int b = 0; b < kBatch; ++b) pv[b] = p0 + b < hi ? get(p0 + b) : make_float2(-INFINITY, 0.f);
    merge_partials(M, W, X, pv);
  }
}
// Two threads merge a row, hp = 0 and 1 (M, W, X: its half): s.lse of the tile's rows, and the entropies where `ent` is given.
template <int D>
__device__ __forceinline__ void row_lse(SimtShared<D>& s, bool valid, float M, float W, float X, float* ent) {
  const int r = threadIdx.x & (kSmRows - 1), hp = threadIdx.x / kSmRows;
  const float lw = __log2f(W);
  if (hp == 1) s.half[r] = W > 0.f ? make_float2(M + lw, lw + X / W) : make_float2(-INFINITY, 0.f);
  __syncthreads();
  float lse = INFINITY;                                // rows that do not exist: 2^(x - inf) = 0
  if (hp == 0) {
    const float2 o[1] = {s.half[r]};
    merge_partials(M, W, X, o);
    const float lz = __log2f(W);
    if (valid && W > 0.f) lse = M + lz;
    if (ent) *ent = valid && W > 0.f ? kLn2 * (lz + X / W) : 0.f;
  }
  __syncthreads();
  if (hp == 0) s.lse[r] = lse;
  __syncthreads();
}
// Column sums of a tile over groups of eight rows, to s.col.
template <int D>
__device__ __forceinline__ void sum_columns(const SimtArgs& a, SimtShared<D>& s, const float (&acc)[8][4], int rt, int j0, float c2) {
  const int tr = threadIdx.x >> 4, tc = threadIdx.x & 15;
  float sum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int i = (rt * kSmRows + tr * 8 + q) & (a.w_pad - 1), t_pos = a.N - a.w + i;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float pe = fast_exp2(fmaf(acc[q][c], c2, -s.lse[tr * 8 + q]));
      sum[c] += j0 + tc * 4 + c <= t_pos ? pe : 0.f;
    }
  }
  *reinterpret_cast<float4*>(&s.col[tr][tc * 4]) = make_float4(sum[0], sum[1], sum[2], sum[3]);
  __syncthreads();
}

// Pass 1.  grid = (parts, row tiles x groups, layers): statistics of 128 rows over one key segment.
template <typename T, int D>
__global__ void __launch_bounds__(kSmThreads) simt_pass1(const __grid_constant__ SimtArgs a) {
  extern __shared__ __align__(16) unsigned char simt_smem[];
  SimtShared<D>& s = *reinterpret_cast<SimtShared<D>*>(simt_smem);
  pdl_trigger();
  pdl_wait();
  const int part = blockIdx.x, g = blockIdx.y / a.n_rt, rt = blockIdx.y - g * a.n_rt, layer = blockIdx.z;
  const int tr = threadIdx.x >> 4, tc = threadIdx.x & 15;
  const T* kg = (const T*)a.k[layer] + (size_t)g * a.sh;
  const float c2 = a.c2[layer];
  stage_rows<T, D>(a, (const T*)a.q[layer], g, rt, s.q);
  RowStat st[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) st[r] = RowStat{-INFINITY, 0.f, 0.f};
  const int t_lo = (int)((long long)part * a.n_keys_tiles / a.parts), t_hi = (int)((long long)(part + 1) * a.n_keys_tiles / a.parts);
  for (int t = t_lo; t < t_hi; ++t) {
    const int j0 = t * kSmKeys;
    stage_keys<T, D>(a, kg, j0, s.k);
    __syncthreads();
    float acc[8][4];
    multiply<D>(s, tr, tc, acc);
    __syncthreads();
    add_tile(a, acc, rt, j0, c2, st);
  }
  fold_rows(st, [&](int r, const float2& p) {
    const int row = rt * kSmRows + tr * 8 + r;
    if (row < a.rows_pg_pad) a.part[((size_t)layer * a.parts + part) * a.rows_pad + g * a.rows_pg_pad + row] = p;
  });
}

// Pass 2.  grid = (key tiles, row tiles x groups, layers): merges the rows' partials, then
// cols[h][j] = (1/w) sum_i 2^(x_ij - lse_i) for the heads of 128 rows (a head of 256 rows takes two tiles).
template <typename T, int D>
__global__ void __launch_bounds__(kSmThreads) simt_pass2(const __grid_constant__ SimtArgs a) {
  extern __shared__ __align__(16) unsigned char simt_smem[];
  SimtShared<D>& s = *reinterpret_cast<SimtShared<D>*>(simt_smem);
  pdl_trigger();
  const int span = a.w_pad > kSmRows ? a.w_pad / kSmRows : 1, n_rs = a.n_rt / span;   // row tiles a block takes
  const int j0 = blockIdx.x * kSmKeys, g = blockIdx.y / n_rs, rs = blockIdx.y - g * n_rs, layer = blockIdx.z;
  const int tr = threadIdx.x >> 4, tc = threadIdx.x & 15;
  const float c2 = a.c2[layer];
  pdl_wait();
  if (j0 == 0 && rs == n_rs - 1)                        // rows of the group's last block that no tile holds
    for (int row = a.n_rt * kSmRows + threadIdx.x; row < a.rows_pg_pad; row += kSmThreads)
      a.row_ent[(size_t)layer * a.rows_pad + g * a.rows_pg_pad + row] = 0.f;
  stage_keys<T, D>(a, (const T*)a.k[layer] + (size_t)g * a.sh, j0, s.k);
  float total = 0.f;                                   // heads longer than a tile
  for (int m = 0; m < span; ++m) {
    const int rt = rs * span + m;
    stage_rows<T, D>(a, (const T*)a.q[layer], g, rt, s.q);
    // two threads per row, each half of the partials
    const int r = threadIdx.x & (kSmRows - 1), hp = threadIdx.x / kSmRows, row = rt * kSmRows + r;
    const int p_lo = hp * a.parts / 2, p_hi = (hp + 1) * a.parts / 2;
    float M = -INFINITY, W = 0.f, X = 0.f;
    const bool valid = row < a.rows_pg && (row & (a.w_pad - 1)) < a.w;
    if (valid)
      merge_range(p_lo, p_hi, M, W, X, [&](int p) {
        return __ldcg(a.part + ((size_t)layer * a.parts + p) * a.rows_pad + g * a.rows_pg_pad + row);
      });
    row_lse(s, valid, M, W, X,
            j0 == 0 && row < a.rows_pg_pad ? a.row_ent + (size_t)layer * a.rows_pad + g * a.rows_pg_pad + row : nullptr);
    float acc[8][4];
    multiply<D>(s, tr, tc, acc);
    sum_columns(a, s, acc, rt, j0, c2);
    // sums over a head's groups of eight rows
    const int per_head = min(a.w_pad, kSmRows) / 8, heads = kSmRows / 8 / per_head;
    for (int x = threadIdx.x; x < heads * kSmKeys; x += kSmThreads) {
      const int hh = x / kSmKeys, j = x % kSmKeys;
      float t = 0.f;
      for (int e = 0; e < per_head; ++e) t += s.col[hh * per_head + e][j];
      total += t;
      const int head = (rt * kSmRows) / a.w_pad + hh;
      if (m == span - 1 && head < a.group && j0 + j < a.N)
        a.cols[(size_t)layer * a.cols_layer_stride + (size_t)(g * a.group + head) * a.col_stride + j0 + j] =
            (span > 1 ? total : t) / (float)a.w;
    }
    __syncthreads();
  }
}

// Both passes of a short call at once (at most kSimtParts key tiles, heads of at most 128 rows): grid = (key tiles, row tiles x
// groups, layers), and all blocks run at the same time.  A block keeps its 128 x 64 logits in registers while the blocks of
// its rows exchange their partials, the same ones and merged the same way: the bits of the two passes.  What it
// saves is the second staging and multiplication, and a launch.  8 heads, window 32, head dim 64, us with the sums over heads,
// two passes / this: 4 layers of 2048 keys 39.5 / 30.1, one layer of 4096 40.5 / 25.8, 2 layers of 700 25.3 / 18.1.
template <typename T, int D>
__global__ void __launch_bounds__(kSmThreads, 3) simt_once(const __grid_constant__ SimtArgs a) {
  extern __shared__ __align__(16) unsigned char simt_smem[];
  SimtShared<D>& s = *reinterpret_cast<SimtShared<D>*>(simt_smem);
  __shared__ int last;
  __shared__ unsigned tag_s;
  pdl_trigger();
  pdl_wait();
  // (one thread reads it: the line is every block's)
  if (threadIdx.x == 0) tag_s = (unsigned)__ldcg(a.ctl + kCtlTag) + 1u;
  const int part = blockIdx.x, g = blockIdx.y / a.n_rt, rt = blockIdx.y - g * a.n_rt, layer = blockIdx.z, j0 = part * kSmKeys;
  const int tr = threadIdx.x >> 4, tc = threadIdx.x & 15;
  const float c2 = a.c2[layer];
  constexpr size_t kEntWords = kXchPairs;
  unsigned long long* const words = a.xch + (size_t)(blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x * kSmRows;   // of these rows: [part][row]
  stage_rows<T, D>(a, (const T*)a.q[layer], g, rt, s.q);
  stage_keys<T, D>(a, (const T*)a.k[layer] + (size_t)g * a.sh, j0, s.k);
  __syncthreads();
  const unsigned tag = tag_s;
  float acc[8][4];
  multiply<D>(s, tr, tc, acc);
  {
    RowStat st[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) st[r] = RowStat{-INFINITY, 0.f, 0.f};
    add_tile(a, acc, rt, j0, c2, st);
    fold_rows(st, [&](int r, const float2& p) {
      unsigned long long* const to = words + part * kSmRows + tr * 8 + r;
      put_word(to, tagged(p.x, tag));
      put_word(to + kEntWords, tagged(p.y, tag));
    });
  }
  float* const ent = a.row_ent + (size_t)layer * a.rows_pad + g * a.rows_pg_pad;
  if (part == 0 && rt == a.n_rt - 1)                    // rows of the group's last block that no tile holds
    for (int row = a.n_rt * kSmRows + threadIdx.x; row < a.rows_pg_pad; row += kSmThreads) ent[row] = 0.f;
  const int r = threadIdx.x & (kSmRows - 1), hp = threadIdx.x / kSmRows, row = rt * kSmRows + r;
  const int p_lo = hp * a.parts / 2, p_hi = (hp + 1) * a.parts / 2;
  float M = -INFINITY, W = 0.f, X = 0.f;
  const bool valid = row < a.rows_pg && (row & (a.w_pad - 1)) < a.w;
  if (valid) {
    // all of the row's words are there, or the wait's bound expires
    long long t0 = 0;
    for (bool all = false; !all;) {
      all = true;
#pragma unroll 8
      for (int p = p_lo; p < p_hi; ++p) {
        const unsigned long long x = get_word(words + p * kSmRows + r), y = get_word(words + p * kSmRows + r + kEntWords);
        all = all && word_has(x, tag) && word_has(y, tag);
      }
      if (all) break;
      const long long now = clock64();
      if (t0 == 0) t0 = now;
      if ((unsigned long long)(now - t0) > kWaitCycles) {
        atomicCAS(a.status, 0, (int)STRUCTKV_ERR_TIMEOUT);
        break;
      }
    }
    merge_range(p_lo, p_hi, M, W, X, [&](int p) {
      return make_float2(word_value(get_word(words + p * kSmRows + r)), word_value(get_word(words + p * kSmRows + r + kEntWords)));
    });
  }
  row_lse(s, valid, M, W, X, part == 0 && row < a.rows_pg_pad ? ent + row : nullptr);
  sum_columns(a, s, acc, rt, j0, c2);
  const int per_head = a.w_pad / 8, heads = kSmRows / 8 / per_head;
  for (int x = threadIdx.x; x < heads * kSmKeys; x += kSmThreads) {
    const int hh = x / kSmKeys, j = x % kSmKeys, head = rt * kSmRows / a.w_pad + hh;
    float t = 0.f;
    for (int e = 0; e < per_head; ++e) t += s.col[hh * per_head + e][j];
    if (head < a.group && j0 + j < a.N)
      a.cols[(size_t)layer * a.cols_layer_stride + (size_t)(g * a.group + head) * a.col_stride + j0 + j] = t / (float)a.w;
  }
  if (threadIdx.x == 0) last = atomicAdd(a.ctl + kCtlExit, 1) == (int)(gridDim.x * gridDim.y * gridDim.z) - 1;
  __syncthreads();
  if (last) pass_tags_on(a.xch, a.ctl, tag, (int)threadIdx.x, (int)blockDim.x);
}

template <typename T, int D>
cudaError_t launch_typed(const Ctx& ctx, const SimtArgs& a, int layers, cudaStream_t st) {
  // Devices whose shared-memory limits have been raised, and the blocks of the one launch an SM of theirs holds.
  static std::atomic<unsigned long long> ready{0};
  static std::atomic<int> per_sm[64];
  const int dev = ctx.device & 63, smem = (int)sizeof(SimtShared<D>);
  const unsigned long long bit = 1ull << dev;
  if (!(ready.load(std::memory_order_acquire) & bit)) {
    int n = 0;
    cudaError_t e = cudaFuncSetAttribute(simt_pass1<T, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(simt_pass2<T, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(simt_once<T, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, simt_once<T, D>, kSmThreads, smem);
    if (e != cudaSuccess) return e;
    per_sm[dev].store(n, std::memory_order_relaxed);
    ready.fetch_or(bit, std::memory_order_release);
  }
  const int G = ctx.cfg.n_kv_heads, span = a.w_pad > kSmRows ? a.w_pad / kSmRows : 1;
  // The layers whose blocks all run at once, as even as it goes (8 layers of 4096 keys: 110 us in two passes, 89
  // three layers at a time; 32 of 2048 keys 187 / 160).
  const long long per_layer = (long long)a.n_keys_tiles * a.n_rt * G;
  const int room = (int)(std::min((long long)per_sm[dev].load(std::memory_order_relaxed) * ctx.sm_count, (long long)kXchPairs / kSmRows) / per_layer);
  if (span == 1 && a.n_keys_tiles == a.parts && room >= 1) {
    const int launches = (layers + room - 1) / room;
    cudaError_t e = clean_words(ctx, st);
    for (int i = 0; i < launches && e == cudaSuccess; ++i) {
      const int lo = i * layers / launches, n = (i + 1) * layers / launches - lo;
      SimtArgs b = a;
      for (int l = 0; l < n; ++l) { b.q[l] = a.q[lo + l]; b.k[l] = a.k[lo + l]; b.c2[l] = a.c2[lo + l]; }
      b.row_ent += (size_t)lo * a.rows_pad;
      b.cols += (size_t)lo * a.cols_layer_stride;
      e = launch_cooperative(simt_once<T, D>, dim3(a.n_keys_tiles, a.n_rt * G, n), dim3(kSmThreads), smem, st, b);
    }
    // where the device does not give this process all of its SMs at once, the two passes do it
    if (e != cudaErrorCooperativeLaunchTooLarge) return e;
    cudaGetLastError();
  }
  const cudaError_t e = launch_pdl(simt_pass1<T, D>, dim3(a.parts, a.n_rt * G, layers), dim3(kSmThreads), smem, st, a);
  if (e != cudaSuccess) return e;
  return launch_pdl(simt_pass2<T, D>, dim3(a.n_keys_tiles, a.n_rt / span * G, layers), dim3(kSmThreads), smem, st, a);
}

}  // namespace

size_t simt_part_entries(const structkv_config& cfg, int n) {
  const size_t rows = align_up((size_t)(cfg.n_q_heads / cfg.n_kv_heads) * tc_window_pad(cfg.window), kRowBlock) * cfg.n_kv_heads;
  return (size_t)std::min(n, kSmLayers) * kSimtParts * rows;
}

cudaError_t launch_score_simt(const Ctx& ctx, const ScoreCall& c, cudaStream_t st) {
  SimtArgs a = {};
  a.sh = c.k_stride_head; a.st = c.k_stride_token;
  a.N = c.n_keys; a.w = ctx.cfg.window; a.w_pad = ctx.w_pad;
  while (1 << a.w_shift < a.w_pad) ++a.w_shift;
  a.group = ctx.cfg.n_q_heads / ctx.cfg.n_kv_heads;
  a.rows_pg = a.group * a.w_pad; a.rows_pg_pad = ctx.rows_pad / ctx.cfg.n_kv_heads; a.rows_pad = ctx.rows_pad;
  // row tiles that hold rows, an even number where a head takes two
  a.n_rt = (a.rows_pg + kSmRows - 1) / kSmRows;
  a.n_keys_tiles = (a.N + kSmKeys - 1) / kSmKeys;
  a.parts = std::min(a.n_keys_tiles, kSimtParts);
  a.xch = ctx.ws.xch; a.ctl = ctx.ws.ctl; a.status = ctx.ws.status;
  a.part = c.part; a.col_stride = c.col_stride; a.cols_layer_stride = c.cols_layer_stride;
  for (int l0 = 0; l0 < c.n; l0 += kSmLayers) {
    const int layers = std::min(kSmLayers, c.n - l0);
    for (int l = 0; l < layers; ++l) {
      a.q[l] = c.q[l0 + l]; a.k[l] = c.k[l0 + l];
      a.c2[l] = c.scale[l0 + l] * kLog2e;
    }
    a.row_ent = c.row_ent + (size_t)l0 * ctx.rows_pad;
    a.cols = c.cols + (size_t)l0 * c.cols_layer_stride;
    const bool f32 = ctx.cfg.dtype == STRUCTKV_FP32;
    cudaError_t e = cudaErrorInvalidValue;
    if (ctx.cfg.head_dim == 64) e = f32 ? launch_typed<float, 64>(ctx, a, layers, st) : launch_typed<__nv_bfloat16, 64>(ctx, a, layers, st);
    if (ctx.cfg.head_dim == 128) e = f32 ? launch_typed<float, 128>(ctx, a, layers, st) : launch_typed<__nv_bfloat16, 128>(ctx, a, layers, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace skv
