// stage_f64t.cu -- stage-kernel instantiations: FP64 path, Cartesian Euler blocks, the second
// tile height the group tuner may choose, and stages 1 and 2 with the halo exchange folded in
// (both heights) (TY_ALT_F64)
#include <atomic>

#include "launch.h"
#include "stage_x.cuh"

namespace gbcfd {
cudaError_t launch_stage_f64_alt(int stage, const GroupParams& P, int grid, cudaStream_t s) {
  return xstage_dispatch<false, false, TY_ALT_F64>(stage, P, grid, s);
}
cudaError_t stage_prepare_f64_alt() { return xstage_prepare<false, false, TY_ALT_F64>(); }
int stage_occupancy_f64_alt() { return 1; }
cudaError_t launch_stage_f64_push(int stage, int ty, const GroupParams& P, int grid, cudaStream_t s) {
  if (ty == TY_ALT_F64) return xstage_dispatch_push<TY_ALT_F64>(stage, P, grid, s);
  if (ty == TY_DEFAULT) return xstage_dispatch_push<TY_DEFAULT>(stage, P, grid, s);
  return cudaErrorInvalidValue;
}
cudaError_t stage_prepare_f64_push(int ty) {
  if (ty == TY_ALT_F64) return xstage_prepare_push<TY_ALT_F64>();
  if (ty == TY_DEFAULT) return xstage_prepare_push<TY_DEFAULT>();
  return cudaErrorInvalidValue;
}
}  // namespace gbcfd
