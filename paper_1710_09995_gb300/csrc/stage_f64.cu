// stage_f64.cu -- stage-kernel instantiations: FP64 path, Cartesian grids
#include <atomic>

#include "launch.h"
#include "stage_x.cuh"

namespace gbcfd {
cudaError_t launch_stage_f64(int viscous, int stage, const GroupParams& P, int grid,
                             cudaStream_t s) {
  return viscous ? xstage_dispatch<true, false, TY_DEFAULT>(stage, P, grid, s)
                 : xstage_dispatch<false, false, TY_DEFAULT>(stage, P, grid, s);
}
cudaError_t stage_prepare_f64(int viscous) {
  return viscous ? xstage_prepare<true, false, TY_DEFAULT>() : xstage_prepare<false, false, TY_DEFAULT>();
}
int stage_occupancy_f64(int) { return 1; }  // one CTA fills an SM's registers and shared memory
}  // namespace gbcfd
