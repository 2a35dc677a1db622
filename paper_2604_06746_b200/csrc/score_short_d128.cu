// Scorer of one layer of few keys, head dimension 128.
#include "score_short.cuh"

namespace skv {
cudaError_t short_launch_128(int shape, const ShortParams& p, int grid, int device, cudaStream_t st) {
  return short_dispatch<128>(shape, p, grid, device, st);
}
}  // namespace skv
