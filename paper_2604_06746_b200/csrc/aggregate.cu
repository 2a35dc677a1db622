// Block-level aggregation of token scores for block-based KV memory managers, and the
// attention-mass recovery diagnostic.  Both are fixed-order fp32 reductions (deterministic).
#include "radix.cuh"

namespace skv {
namespace {

// One thread per block of `block_size` consecutive tokens: S_block_k = sum_{t in block k} score[t].
// The last block of a vector may be ragged.
__global__ void block_scores(const float* __restrict__ scores, long long row_stride, int n,
                             int block_size, int n_blocks, int vec4, float* __restrict__ out) {
  pdl_trigger();
  pdl_wait();
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n_blocks) return;
  const float* s = scores + (size_t)blockIdx.y * row_stride;
  const int lo = k * block_size, hi = min(n, lo + block_size);
  float acc = 0.f;
  if (vec4 && hi - lo == block_size) {                   // whole block, 16-byte loads, same token order
    const float4* s4 = reinterpret_cast<const float4*>(s + lo);
#pragma unroll 4
    for (int q = 0; q < block_size / 4; ++q) {
      const float4 v = s4[q];
      acc += v.x; acc += v.y; acc += v.z; acc += v.w;
    }
  } else {
    for (int t = lo; t < hi; ++t) acc += s[t];
  }
  out[(size_t)blockIdx.y * n_blocks + k] = acc;
}

// out[g][j] = sum of the pooled attention of the `group` query heads that share KV head g, heads
// in ascending order.
template <typename T>
__global__ void __launch_bounds__(256)
group_saliency(const float* __restrict__ head_cols, long long col_stride, int group, int n, float* __restrict__ out) {
  pdl_trigger();
  pdl_wait();
  const int j = (blockIdx.x * blockDim.x + threadIdx.x) * (int)(sizeof(T) / sizeof(float));
  if (j >= n) return;
  const int g = blockIdx.y;
  T acc{};
#pragma unroll 4
  for (int q = 0; q < group; ++q)
    add_to(acc, *reinterpret_cast<const T*>(head_cols + (size_t)(g * group + q) * col_stride + j));
  *reinterpret_cast<T*>(out + (size_t)g * n + j) = acc;
}

__device__ __forceinline__ float block_sum(float v, float* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) red[warp] = v;
  __syncthreads();
  if (warp == 0) {
    v = red[lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  }
  return v;
}

// A cluster of CL CTAs per score vector: out = (sum of the scores at idx) / (sum of all scores), each
// CTA a slice of both, the slices added in order.  An index outside [0, n) contributes nothing and is
// recorded in the status word.  Bound by reading the scores; one CTA per vector left 116 SMs idle and
// one load in flight per thread (32 vectors of 131072: 20 us).
template <int CL>
__global__ void __launch_bounds__(kRxThreads)
mass_recovery(const float* __restrict__ scores, long long row_stride, int n, const int* __restrict__ idx,
              int n_idx, float* __restrict__ out, int* __restrict__ status) {
  __shared__ float red[2][32];
  __shared__ float slots[2 * CL];
  const int tid = threadIdx.x, rank = CL > 1 ? (int)cg::this_cluster().block_rank() : 0;
  const float* s = scores + (size_t)(blockIdx.x / CL) * row_stride;
  pdl_trigger();
  cluster_barrier<CL>();                             // all CTAs of the cluster run before any remote access
  pdl_wait();
  float kept = 0.f, total = 0.f;
  const int ip = (n_idx + CL - 1) / CL, i_hi = min(n_idx, (rank + 1) * ip);
#pragma unroll 4
  for (int r = rank * ip + tid; r < i_hi; r += kRxThreads) {
    const int j = idx[r];
    if (j >= 0 && j < n) kept += s[j];
    else atomicCAS(status, 0, (int)STRUCTKV_ERR_INVALID_ARG);
  }
  const int per = ((n + CL - 1) / CL + 3) & ~3, lo = min(n, rank * per), hi = min(n, lo + per);
  if (((uintptr_t)s & 15) == 0) {
    const float4* s4 = reinterpret_cast<const float4*>(s + lo);
    const int n4 = (hi - lo) / 4;
#pragma unroll 4
    for (int q = tid; q < n4; q += kRxThreads) {
      const float4 v = s4[q];
      total += (v.x + v.y) + (v.z + v.w);
    }
    for (int j = lo + 4 * n4 + tid; j < hi; j += kRxThreads) total += s[j];
  } else {
#pragma unroll 8
    for (int j = lo + tid; j < hi; j += kRxThreads) total += s[j];
  }
  kept = block_sum(kept, red[0]);
  total = block_sum(total, red[1]);
  if (CL > 1) {
    if (tid == 0) {
      float* to = cg::this_cluster().map_shared_rank(slots, 0);
      to[2 * rank] = kept;
      to[2 * rank + 1] = total;
    }
    cluster_barrier<CL>();
    if (rank == 0 && tid == 0) {
      kept = total = 0.f;
      for (int r = 0; r < CL; ++r) { kept += slots[2 * r]; total += slots[2 * r + 1]; }
    }
  }
  if (rank == 0 && tid == 0) out[blockIdx.x / CL] = kept / total;
}

}  // namespace

cudaError_t launch_block_scores(const float* scores, long long row_stride, int batch, int n, int block_size,
                                float* out, cudaStream_t st) {
  const int n_blocks = (n + block_size - 1) / block_size;
  const int vec4 = (block_size % 4 == 0) && ((uintptr_t)scores % 16 == 0) && (batch == 1 || row_stride % 4 == 0);
  return launch_pdl(block_scores, dim3((n_blocks + 127) / 128, batch), dim3(128), 0, st, scores, row_stride, n,
                    block_size, n_blocks, vec4, out);
}

cudaError_t launch_group_saliency(const float* head_cols, long long col_stride, int n_heads, int group, int n,
                                  float* out, cudaStream_t st) {
  if (n % 4 == 0 && col_stride % 4 == 0 && (uintptr_t)head_cols % 16 == 0 && (uintptr_t)out % 16 == 0)
    return launch_pdl(group_saliency<float4>, dim3((n / 4 + 255) / 256, n_heads / group), dim3(256), 0, st, head_cols,
                      col_stride, group, n, out);
  return launch_pdl(group_saliency<float>, dim3((n + 255) / 256, n_heads / group), dim3(256), 0, st, head_cols, col_stride,
                    group, n, out);
}

cudaError_t launch_mass_recovery(const float* scores, long long row_stride, int batch, int n, const int* idx,
                                 int n_idx, float* out, int* status, cudaStream_t st) {
  // a slice below 4096 scores is not worth the exchange
  if (n <= 4096) return launch_cluster<1>(mass_recovery<1>, dim3(batch), dim3(kRxThreads), 0, st, scores, row_stride, n, idx, n_idx, out, status);
  return launch_cluster<8>(mass_recovery<8>, dim3(batch * 8), dim3(kRxThreads), 0, st, scores, row_stride, n, idx, n_idx, out, status);
}

}  // namespace skv
