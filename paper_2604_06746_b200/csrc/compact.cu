// Row gather / compaction: dst[s, r, :] = src[s, idx[r], :], byte exact.  Rows are split into
// 16-byte (or 4-byte / 1-byte) units; consecutive threads take consecutive units of a row, so
// writes are fully coalesced and reads are coalesced within each gathered row.
// Bound by DRAM: 32 layers x 16 slabs x 16384 rows of 256 bytes 690 us, 6.22 TB/s (a plain copy: 6.46); 2048 rows a
// slab 93 us.  With a 64-bit division per unit and blocks striding over the whole output these took 745 and 107: the
// divisions used more issue slots than the loads.  Two, four and eight loads in flight per thread: 690 / 696 / 687 us.
#include "common.cuh"

#include <algorithm>

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

// u / d for u < 2^31 by one multiplication and a shift, after Granlund and Montgomery (Division by Invariant Integers using
// Multiplication, 1994); a 64-bit division took some 100 instructions, two of them per 16 bytes.
struct Divisor { unsigned mul; int shift; };               // mul 0: d is 1
inline Divisor divisor(unsigned d) {
  int l = 0;
  while ((1ull << l) < d) ++l;
  return d == 1 ? Divisor{0, 0} : Divisor{(unsigned)((1ull << (31 + l)) / d + 1), l - 1};
}
__device__ __forceinline__ unsigned operator/(unsigned u, const Divisor& d) {
  return d.mul == 0 ? u : __umulhi(u, d.mul) >> d.shift;
}

// One list's rows out of one slab after the other: block `block` of `blocks`, every `slab_step`-th slab from `slab` on.  A block
// takes kCpUnroll * kCpThreads consecutive units.
struct Gather {
  long long slab_stride, row_stride, idx_slab_stride;
  Divisor per_row;                     // units of a row
  unsigned row_units, units;           // units this launch writes in a slab
  unsigned long long slab_units;       // from slab to slab of the output
  int n_slabs, n_rows_src;
};
template <typename V>
__device__ __forceinline__ void gather_blocks(const Gather& g, unsigned block, unsigned blocks, int slab, int slab_step,
                                              const char* __restrict__ src, const int* __restrict__ idx, char* __restrict__ dst,
                                              int* __restrict__ status) {
  for (int s = slab; s < g.n_slabs; s += slab_step) {
    const char* const from = src + s * g.slab_stride;
    const int* const list = idx + s * g.idx_slab_stride;   // stride 0: one list for every slab
    V* const to = reinterpret_cast<V*>(dst) + s * g.slab_units;
    for (unsigned u0 = block * (kCpThreads * kCpUnroll) + threadIdx.x; u0 < g.units; u0 += blocks * (kCpThreads * kCpUnroll)) {
      V val[kCpUnroll];
      int j[kCpUnroll];
#pragma unroll
      for (int e = 0; e < kCpUnroll; ++e) {
        const unsigned u = u0 + e * kCpThreads;
        j[e] = u < g.units ? __ldg(list + u / g.per_row) : -1;
      }
#pragma unroll
      for (int e = 0; e < kCpUnroll; ++e) {
        const unsigned u = u0 + e * kCpThreads, c = u - u / g.per_row * g.row_units;
        if (j[e] >= 0 && j[e] < g.n_rows_src)
          val[e] = ld_stream(reinterpret_cast<const V*>(from + j[e] * g.row_stride) + c);
        else if (u < g.units && c == 0)
          atomicCAS(status, 0, (int)STRUCTKV_ERR_INVALID_ARG);
      }
#pragma unroll
      for (int e = 0; e < kCpUnroll; ++e)
        if (j[e] >= 0 && j[e] < g.n_rows_src) st_stream(to + u0 + e * kCpThreads, val[e]);
    }
  }
}

template <typename V>
__global__ void __launch_bounds__(kCpThreads)
gather_rows(const Gather g, const char* __restrict__ src, const int* __restrict__ idx, char* __restrict__ dst,
            int* __restrict__ status) {
  pdl_trigger();
  pdl_wait();
  gather_blocks<V>(g, blockIdx.x, gridDim.x, blockIdx.y, gridDim.y, src, idx, dst, status);
}
// Block `block` of one word per row of a second source, by the same list.
__device__ __forceinline__ void gather_words(const CompactWords& w, int block, const int* __restrict__ idx, int n_idx, int n_rows_src) {
  const int r = block * kCpThreads + (int)threadIdx.x;
  if (r >= n_idx) return;
  const int j = __ldg(idx + r);
  if (j >= 0 && j < n_rows_src)
    reinterpret_cast<unsigned*>(w.dst)[r] = *reinterpret_cast<const unsigned*>((const char*)w.src + j * w.row_stride);
}
// The last `words` blocks do that (a launch of its own for 4 bytes a row took 2 to 3 us after the gather it follows: the
// smallest whole prefill 66.8 -> 65.0 us).
template <typename V>
__global__ void __launch_bounds__(kCpThreads)
gather_rows_words(const Gather g, const char* __restrict__ src, const int* __restrict__ idx, int n_idx,
                  char* __restrict__ dst, int* __restrict__ status, const CompactWords w, int words) {
  pdl_trigger();
  pdl_wait();
  const int rows = (int)gridDim.x - words;
  if ((int)blockIdx.x >= rows) gather_words(w, (int)blockIdx.x - rows, idx, n_idx, g.n_rows_src);
  else gather_blocks<V>(g, blockIdx.x, rows, blockIdx.y, gridDim.y, src, idx, dst, status);
}

// The same gather for several layers in one launch: layer blockIdx.z reads its own source (the
// pointers travel as a kernel argument), its own index list and writes its own slabs of dst.
struct LayerPtrs { const char* src[kMaxGatherLayers]; };

template <typename V>
__global__ void __launch_bounds__(kCpThreads)
gather_rows_layers(const Gather g, const __grid_constant__ LayerPtrs srcs, const int* __restrict__ idx,
                   long long idx_layer_stride, char* __restrict__ dst, long long dst_layer_stride, int* __restrict__ status) {
  pdl_trigger();
  pdl_wait();
  const int layer = blockIdx.z;
  gather_blocks<V>(g, blockIdx.x, gridDim.x, blockIdx.y, gridDim.y, srcs.src[layer], idx + (long long)layer * idx_layer_stride,
                   dst + (long long)layer * dst_layer_stride, status);
}
// The same, and one slab of another source by another list, with a word per row beside it, in blocks behind the layers': what
// follows the selections of a whole prefill, in one launch (two took 2 us longer: the smallest whole prefill 40.4 -> 37.6 us).
// One dimension of blocks: `blocks` for a slab, then `other_blocks`, then the words'.
struct OtherRows { Gather g; const char* src; const int* idx; char* dst; CompactWords words; int n_idx, blocks; };
template <typename V>
__global__ void __launch_bounds__(kCpThreads)
gather_rows_prefill(const Gather g, const __grid_constant__ LayerPtrs srcs, const int* __restrict__ idx, long long idx_layer_stride,
                    char* __restrict__ dst, long long dst_layer_stride, int* __restrict__ status, int n_layers, int blocks,
                    const __grid_constant__ OtherRows o) {
  pdl_trigger();
  pdl_wait();
  const int per_layer = blocks * g.n_slabs, b = (int)blockIdx.x - n_layers * per_layer;
  if (b < 0) {
    const int layer = (int)blockIdx.x / per_layer, in = (int)blockIdx.x - layer * per_layer, slab = in / blocks;
    gather_blocks<V>(g, in - slab * blocks, blocks, slab, g.n_slabs, srcs.src[layer], idx + (long long)layer * idx_layer_stride,
                     dst + (long long)layer * dst_layer_stride, status);
  } else if (b < o.blocks) {
    gather_blocks<uint4>(o.g, b, o.blocks, 0, 1, o.src, o.idx, o.dst, status);
  } else {
    gather_words(o.words, b - o.blocks, o.idx, o.n_idx, o.g.n_rows_src);
  }
}

// The unit of a copy whose pointers, strides and row size have the low bits `low` between them, and the launch over it: at
// most kCpBlocksPerSm blocks an SM.  A launch counts its units of a slab in 31 bits: longer lists go `rows` at a time.
struct Plan {
  Gather g;
  int unit, rows;
  dim3 grid;
  Plan(unsigned long long low, long long slab_stride, long long row_stride, int row_bytes, int n_slabs, int n_rows_src,
       long long idx_slab_stride, int n_idx)
      : unit(low % 16 == 0 ? 16 : low % 4 == 0 ? 4 : 1) {
    const unsigned per_row = (unsigned)(row_bytes / unit);
    g = Gather{slab_stride, row_stride, idx_slab_stride, divisor(per_row), per_row, 0, (unsigned long long)per_row * n_idx, n_slabs, n_rows_src};
    rows = (int)std::min((long long)n_idx, 0x7fffffffll / per_row);
  }
  void take(int n, int n_layers, int sm_count) {           // the next n indices
    g.units = (unsigned)n * g.row_units;
    const long long want = ((long long)g.units + kCpThreads * kCpUnroll - 1) / (kCpThreads * kCpUnroll);
    const long long slabs = std::min(g.n_slabs, 32768), cap = (long long)sm_count * kCpBlocksPerSm / (slabs * n_layers);
    grid = dim3((unsigned)std::max(1ll, std::min(want, cap)), (unsigned)slabs, (unsigned)n_layers);
  }
};

}  // namespace

bool launch_compact_prefill(const CompactRows& kv, const void* const* srcs, int n_layers, long long idx_layer_stride,
                            long long dst_layer_stride, const CompactRows& other, const CompactWords& words, int* status, int sm_count,
                            cudaStream_t st, cudaError_t* e) {
  LayerPtrs lp;
  unsigned long long low = (uintptr_t)kv.dst | kv.slab_stride | kv.row_stride | kv.row_bytes | dst_layer_stride;
  for (int l = 0; l < n_layers; ++l) {
    lp.src[l] = (const char*)srcs[l];
    low |= (uintptr_t)srcs[l];
  }
  Plan p(low, kv.slab_stride, kv.row_stride, kv.row_bytes, kv.n_slabs, kv.n_rows_src, 0, kv.n_idx);
  Plan q((uintptr_t)other.src | (uintptr_t)other.dst | other.row_stride | other.row_bytes, 0, other.row_stride, other.row_bytes, 1,
         other.n_rows_src, 0, other.n_idx);
  if (kv.n_idx < 1 || kv.n_slabs < 1 || n_layers < 1 || other.n_idx < 1 || p.unit != 16 || q.unit != 16 || p.rows < kv.n_idx ||
      q.rows < other.n_idx)
    return false;
  p.take(kv.n_idx, n_layers, sm_count);
  q.take(other.n_idx, 1, sm_count);
  const long long first = (long long)p.grid.x * kv.n_slabs * n_layers, last = (other.n_idx + kCpThreads - 1) / kCpThreads;
  if (first + q.grid.x + last > 0x7fffffffll) return false;
  const OtherRows o = {q.g, (const char*)other.src, other.idx, (char*)other.dst, words, other.n_idx, (int)q.grid.x};
  *e = launch_pdl(gather_rows_prefill<uint4>, dim3((unsigned)(first + q.grid.x + last)), dim3(kCpThreads), 0, st, p.g, lp, kv.idx,
                  idx_layer_stride, (char*)kv.dst, dst_layer_stride, status, n_layers, (int)p.grid.x, o);
  return true;
}

cudaError_t launch_compact_layers(const void* const* srcs, int n_layers, long long slab_stride, long long row_stride,
                                  int row_bytes, int n_slabs, int n_rows_src, const int* idx,
                                  long long idx_layer_stride, int n_idx, void* dst, long long dst_layer_stride,
                                  int* status, int sm_count, cudaStream_t st) {
  if (n_idx == 0 || n_slabs == 0 || n_layers == 0) return cudaSuccess;
  LayerPtrs lp;
  unsigned long long low = (uintptr_t)dst | slab_stride | row_stride | row_bytes | dst_layer_stride;
  for (int l = 0; l < n_layers; ++l) {
    lp.src[l] = (const char*)srcs[l];
    low |= (uintptr_t)srcs[l];
  }
  Plan p(low, slab_stride, row_stride, row_bytes, n_slabs, n_rows_src, 0, n_idx);
  const auto kernel = p.unit == 16 ? gather_rows_layers<uint4> : p.unit == 4 ? gather_rows_layers<unsigned> : gather_rows_layers<unsigned char>;
  for (int r = 0; r < n_idx; r += p.rows) {
    p.take(std::min(p.rows, n_idx - r), n_layers, sm_count);
    const cudaError_t e = launch_pdl(kernel, p.grid, dim3(kCpThreads), 0, st, p.g, lp, idx + r, idx_layer_stride,
                                     (char*)dst + (long long)r * row_bytes, dst_layer_stride, status);
    if (e != cudaSuccess || n_idx - r <= p.rows) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_compact(const void* src, long long slab_stride, long long row_stride,
                           int row_bytes, int n_slabs, int n_rows_src, const int* idx,
                           long long idx_slab_stride, int n_idx, void* dst, int* status, int sm_count,
                           cudaStream_t st, const CompactWords* words) {
  if (n_idx == 0 || n_slabs == 0) return cudaSuccess;
  Plan p((uintptr_t)src | (uintptr_t)dst | slab_stride | row_stride | row_bytes, slab_stride, row_stride, row_bytes, n_slabs, n_rows_src,
         idx_slab_stride, n_idx);
  const auto both = p.unit == 16 ? gather_rows_words<uint4> : p.unit == 4 ? gather_rows_words<unsigned> : gather_rows_words<unsigned char>;
  const auto kernel = p.unit == 16 ? gather_rows<uint4> : p.unit == 4 ? gather_rows<unsigned> : gather_rows<unsigned char>;
  for (int r = 0; r < n_idx; r += p.rows) {
    p.take(std::min(p.rows, n_idx - r), 1, sm_count);
    char* const to = (char*)dst + (long long)r * row_bytes;
    cudaError_t e;
    if (words && r == 0) {
      const unsigned extra = ((unsigned)n_idx + kCpThreads - 1) / kCpThreads;
      e = launch_pdl(both, dim3(p.grid.x + extra), dim3(kCpThreads), 0, st, p.g, (const char*)src, idx, n_idx, to, status, *words,
                     (int)extra);
    } else {
      e = launch_pdl(kernel, p.grid, dim3(kCpThreads), 0, st, p.g, (const char*)src, idx + r, to, status);
    }
    if (e != cudaSuccess || n_idx - r <= p.rows) return e;
  }
  return cudaSuccess;
}

}  // namespace skv
