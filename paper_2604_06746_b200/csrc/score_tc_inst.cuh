// Instantiates the tensor-core scorer for one head dimension and parameter size.
#include "score_tc.cuh"

namespace skv {
namespace {
template <int D, int MAXP>
cudaError_t tc_dispatch(int shape, const TcParams<MAXP>& p, int grid, int device, cudaStream_t st) {
  switch (shape) {
    case kWide16: return tc_launch<D, kWide16, MAXP>(p, grid, device, st);
    case kWide32: return tc_launch<D, kWide32, MAXP>(p, grid, device, st);
    case kWide64: return tc_launch<D, kWide64, MAXP>(p, grid, device, st);
    case kWide128: return tc_launch<D, kWide128, MAXP>(p, grid, device, st);
    case kWide256: return tc_launch<D, kWide256, MAXP>(p, grid, device, st);
    case kNarrow32: return tc_launch<D, kNarrow32, MAXP>(p, grid, device, st);
    case kNarrow64: return tc_launch<D, kNarrow64, MAXP>(p, grid, device, st);
  }
  return cudaErrorInvalidValue;
}
}  // namespace
}  // namespace skv
