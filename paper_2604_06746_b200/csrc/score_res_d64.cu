// Resident scorer kernels of head dimension 64.
#include "score_res.cuh"

namespace skv {
cudaError_t res_launch_64(const ResParams<1>& p, int device, cudaStream_t st) { return res_launch<64>(p, device, st); }
cudaError_t res_launch_64(const ResParams<kMaxBatch>& p, int device, cudaStream_t st) { return res_launch<64>(p, device, st); }
}  // namespace skv
