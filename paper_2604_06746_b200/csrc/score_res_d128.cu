// Resident scorer kernels of head dimension 128.
#include "score_res.cuh"

namespace skv {
cudaError_t res_launch_128(const ResParams<1>& p, int device, cudaStream_t st) { return res_launch<128>(p, device, st); }
cudaError_t res_launch_128(const ResParams<kMaxBatch>& p, int device, cudaStream_t st) { return res_launch<128>(p, device, st); }
}  // namespace skv
