// Tensor-core scorer, head dimension 128, one problem per launch.
#include "score_tc_inst.cuh"

namespace skv {
cudaError_t tc_launch_128(int shape, const TcParams<1>& p, int grid, int device, cudaStream_t st) {
  return tc_dispatch<128, 1>(shape, p, grid, device, st);
}
}  // namespace skv
