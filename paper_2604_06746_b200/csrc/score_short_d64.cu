// Scorer of one layer of few keys, head dimension 64.
#include "score_short.cuh"

namespace skv {
cudaError_t short_launch_64(int shape, const ShortParams& p, int grid, int device, cudaStream_t st) {
  return short_dispatch<64>(shape, p, grid, device, st);
}
}  // namespace skv
