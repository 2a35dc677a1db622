// Row gather / compaction: dst[s, r, :] = src[s, idx[r], :], byte exact.  Rows are split into
// 16-byte (or 4-byte / 1-byte) units; consecutive threads take consecutive units of a row, so
// writes are fully coalesced and reads are coalesced within each gathered row.  Two loads in
// flight per thread and up to 64 resident blocks per SM measured best on B200 (more unrolling
// or fewer, fatter blocks lose 10-25 % of the copy bandwidth).
#include "common.cuh"

namespace skv {
namespace {

constexpr int kCpThreads = 256, kCpUnroll = 2, kCpBlocksPerSm = 64;

// Rows are read once and written once: loads bypass L1 allocation, stores are streaming.
template <typename V> __device__ __forceinline__ V ld_stream(const V* p) { return *p; }
template <typename V> __device__ __forceinline__ void st_stream(V* p, const V& v) { *p = v; }
template <> __device__ __forceinline__ uint4 ld_stream<uint4>(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
template <> __device__ __forceinline__ void st_stream<uint4>(uint4* p, const uint4& v) {
  asm volatile("st.global.cs.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// Block 0 .. blocks - 1 of a gather.
template <typename V>
__device__ __forceinline__ void
gather_blocks(int blocks, const char* __restrict__ src, long long slab_stride, long long row_stride,
              int units_per_row, int n_slabs, int n_rows_src, const int* __restrict__ idx,
              long long idx_slab_stride, int n_idx,
              char* __restrict__ dst, int* __restrict__ status) {
  const long long total = (long long)n_slabs * n_idx * units_per_row;
  const long long stride = (long long)blocks * kCpThreads;
  for (long long u0 = (long long)blockIdx.x * kCpThreads + threadIdx.x; u0 < total;
       u0 += stride * kCpUnroll) {
    V val[kCpUnroll];
    bool ok[kCpUnroll];
#pragma unroll
    for (int e = 0; e < kCpUnroll; ++e) {
      const long long u = u0 + e * stride;
      ok[e] = false;
      if (u < total) {
        const long long row = u / units_per_row;           // s * n_idx + r
        const int c = (int)(u - row * units_per_row);
        const int s = (int)(row / n_idx), r = (int)(row - (long long)s * n_idx);
        const int j = __ldg(idx + s * idx_slab_stride + r);   // stride 0: one list for every slab
        if (j >= 0 && j < n_rows_src) {
          val[e] = ld_stream(reinterpret_cast<const V*>(src + s * slab_stride + j * row_stride +
                                                        (long long)c * sizeof(V)));
          ok[e] = true;
        } else if (c == 0) {
          atomicCAS(status, 0, (int)STRUCTKV_ERR_INVALID_ARG);
        }
      }
    }
#pragma unroll
    for (int e = 0; e < kCpUnroll; ++e) {
      const long long u = u0 + e * stride;
      if (ok[e]) st_stream(reinterpret_cast<V*>(dst + u * (long long)sizeof(V)), val[e]);
    }
  }
}

template <typename V>
__global__ void __launch_bounds__(kCpThreads)
gather_rows(const char* __restrict__ src, long long slab_stride, long long row_stride,
            int units_per_row, int n_slabs, int n_rows_src, const int* __restrict__ idx,
            long long idx_slab_stride, int n_idx,
            char* __restrict__ dst, int* __restrict__ status) {
  pdl_trigger();
  pdl_wait();
  gather_blocks<V>(gridDim.x, src, slab_stride, row_stride, units_per_row, n_slabs, n_rows_src, idx, idx_slab_stride, n_idx,
                   dst, status);
}
// The last `words` blocks gather one word per row of a second source by the same list (a launch of its own for
// 4 bytes a row took 2 to 3 us after the gather it follows: the smallest whole prefill 66.8 -> 65.0 us).
template <typename V>
__global__ void __launch_bounds__(kCpThreads)
gather_rows_words(const char* __restrict__ src, long long row_stride, int units_per_row, int n_rows_src,
                  const int* __restrict__ idx, int n_idx, char* __restrict__ dst, int* __restrict__ status,
                  const CompactWords w, int words) {
  pdl_trigger();
  pdl_wait();
  if ((int)blockIdx.x >= (int)gridDim.x - words) {
    const int r = ((int)blockIdx.x - (int)gridDim.x + words) * kCpThreads + (int)threadIdx.x;
    if (r < n_idx) {
      const int j = __ldg(idx + r);
      if (j >= 0 && j < n_rows_src)
        reinterpret_cast<unsigned*>(w.dst)[r] = *reinterpret_cast<const unsigned*>((const char*)w.src + j * w.row_stride);
    }
    return;
  }
  gather_blocks<V>(gridDim.x - words, src, 0, row_stride, units_per_row, 1, n_rows_src, idx, 0, n_idx, dst, status);
}

// The same gather for several layers in one launch: layer blockIdx.y reads its own source (the
// pointers travel as a kernel argument), its own index list and writes its own slab of dst.
struct LayerPtrs { const char* src[kMaxGatherLayers]; };

template <typename V>
__global__ void __launch_bounds__(kCpThreads)
gather_rows_layers(const __grid_constant__ LayerPtrs srcs, long long slab_stride, long long row_stride,
                   int units_per_row, int n_slabs, int n_rows_src, const int* __restrict__ idx,
                   long long idx_layer_stride, int n_idx, char* __restrict__ dst, long long dst_layer_stride,
                   int* __restrict__ status) {
  pdl_trigger();
  pdl_wait();
  const int layer = blockIdx.y;
  gather_blocks<V>(gridDim.x, srcs.src[layer], slab_stride, row_stride, units_per_row, n_slabs, n_rows_src,
                   idx + (long long)layer * idx_layer_stride, 0, n_idx, dst + (long long)layer * dst_layer_stride, status);
}

}  // namespace

cudaError_t launch_compact_layers(const void* const* srcs, int n_layers, long long slab_stride, long long row_stride,
                                  int row_bytes, int n_slabs, int n_rows_src, const int* idx,
                                  long long idx_layer_stride, int n_idx, void* dst, long long dst_layer_stride,
                                  int* status, int sm_count, cudaStream_t st) {
  if (n_idx == 0 || n_slabs == 0 || n_layers == 0) return cudaSuccess;
  LayerPtrs lp;
  bool a16 = ((uintptr_t)dst % 16 == 0) && slab_stride % 16 == 0 && row_stride % 16 == 0 && row_bytes % 16 == 0 &&
             dst_layer_stride % 16 == 0;
  bool a4 = ((uintptr_t)dst % 4 == 0) && slab_stride % 4 == 0 && row_stride % 4 == 0 && row_bytes % 4 == 0 &&
            dst_layer_stride % 4 == 0;
  for (int l = 0; l < n_layers; ++l) {
    lp.src[l] = (const char*)srcs[l];
    a16 = a16 && ((uintptr_t)srcs[l] % 16 == 0);
    a4 = a4 && ((uintptr_t)srcs[l] % 4 == 0);
  }
  const int unit = a16 ? 16 : (a4 ? 4 : 1);
  const int upr = row_bytes / unit;
  const long long total = (long long)n_slabs * n_idx * upr;
  long long blocks = (total + (long long)kCpThreads * kCpUnroll - 1) / ((long long)kCpThreads * kCpUnroll);
  const long long cap = ((long long)sm_count * kCpBlocksPerSm + n_layers - 1) / n_layers;
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  const dim3 grid((unsigned)blocks, (unsigned)n_layers);
  char* d = (char*)dst;
  const auto kernel = unit == 16 ? gather_rows_layers<uint4> : unit == 4 ? gather_rows_layers<unsigned> : gather_rows_layers<unsigned char>;
  return launch_pdl(kernel, grid, dim3(kCpThreads), 0, st, lp, slab_stride, row_stride, upr, n_slabs, n_rows_src, idx,
                    idx_layer_stride, n_idx, d, dst_layer_stride, status);
}

cudaError_t launch_compact(const void* src, long long slab_stride, long long row_stride,
                           int row_bytes, int n_slabs, int n_rows_src, const int* idx,
                           long long idx_slab_stride, int n_idx, void* dst, int* status, int sm_count,
                           cudaStream_t st, const CompactWords* words) {
  if (n_idx == 0 || n_slabs == 0) return cudaSuccess;
  const bool a16 = ((uintptr_t)src % 16 == 0) && ((uintptr_t)dst % 16 == 0) && slab_stride % 16 == 0 &&
                   row_stride % 16 == 0 && row_bytes % 16 == 0;
  const bool a4 = ((uintptr_t)src % 4 == 0) && ((uintptr_t)dst % 4 == 0) && slab_stride % 4 == 0 &&
                  row_stride % 4 == 0 && row_bytes % 4 == 0;
  const int unit = a16 ? 16 : (a4 ? 4 : 1);
  const int upr = row_bytes / unit;
  const long long total = (long long)n_slabs * n_idx * upr;
  long long blocks = (total + (long long)kCpThreads * kCpUnroll - 1) / ((long long)kCpThreads * kCpUnroll);
  const long long cap = (long long)sm_count * kCpBlocksPerSm;
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  const char* s = (const char*)src;
  char* d = (char*)dst;
  if (words) {
    const auto both = unit == 16 ? gather_rows_words<uint4> : unit == 4 ? gather_rows_words<unsigned> : gather_rows_words<unsigned char>;
    const int extra = (n_idx + kCpThreads - 1) / kCpThreads;
    return launch_pdl(both, dim3((unsigned)(blocks + extra)), dim3(kCpThreads), 0, st, s, row_stride, upr, n_rows_src, idx, n_idx,
                      d, status, *words, extra);
  }
  const auto kernel = unit == 16 ? gather_rows<uint4> : unit == 4 ? gather_rows<unsigned> : gather_rows<unsigned char>;
  return launch_pdl(kernel, dim3((unsigned)blocks), dim3(kCpThreads), 0, st, s, slab_stride, row_stride, upr, n_slabs,
                    n_rows_src, idx, idx_slab_stride, n_idx, d, status);
}

}  // namespace skv
