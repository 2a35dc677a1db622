// Tensor-core scorer, head dimension 64, one problem per launch.
#include "score_tc_inst.cuh"

namespace skv {
cudaError_t tc_launch_64(int shape, const TcParams<1>& p, int grid, int device, cudaStream_t st) {
  return tc_dispatch<64, 1>(shape, p, grid, device, st);
}
}  // namespace skv
