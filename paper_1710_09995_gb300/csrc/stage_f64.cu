// stage_f64.cu -- stage-kernel instantiations: FP64 path, Cartesian grids
#include <atomic>

#include "launch.h"
#include "stage_x.cuh"

namespace gbcfd {
cudaError_t launch_stage_f64(int viscous, int stage, const GroupParams& P, int grid,
                             cudaStream_t s) {
  return viscous ? xstage_dispatch<true, TY_DEFAULT>(stage, P, grid, s)
                 : xstage_dispatch<false, TY_DEFAULT>(stage, P, grid, s);
}
cudaError_t stage_prepare_f64(int viscous) {
  return viscous ? xstage_prepare<true, TY_DEFAULT>() : xstage_prepare<false, TY_DEFAULT>();
}
int stage_occupancy_f64(int) { return 1; }  // one CTA fills an SM's registers and shared memory
}  // namespace gbcfd
