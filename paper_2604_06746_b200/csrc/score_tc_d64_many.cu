// Tensor-core scorer, head dimension 64, several problems (layers, sequences) per launch.
#include "score_tc_inst.cuh"

namespace skv {
cudaError_t tc_launch_64(int shape, const TcParams<kMaxBatch>& p, int grid, int device, cudaStream_t st) {
  return tc_dispatch<64, kMaxBatch>(shape, p, grid, device, st);
}
}  // namespace skv
