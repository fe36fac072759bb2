// stage_f64c.cu -- stage-kernel instantiations: FP64 path, curvilinear grids (inviscid blocks with
// the faces on the integer pipes; viscous ones, whose gradients go through the metrics, in FP64)
#include "stage_inst.cuh"
#include "stage_x.cuh"

namespace gbcfd {
cudaError_t launch_stage_f64c(int viscous, int stage, const GroupParams& P, int grid,
                              cudaStream_t s) {
  return viscous ? stage_dispatch_v<double, true, true, TY_DEFAULT>(stage, P, grid, s)
                 : xstage_dispatch<false, true, TY_DEFAULT>(stage, P, grid, s);
}
cudaError_t stage_prepare_f64c(int viscous) {
  return viscous ? stage_prepare_v<double, true, true, TY_DEFAULT>() : xstage_prepare<false, true, TY_DEFAULT>();
}
int stage_occupancy_f64c(int viscous) {
  return viscous ? stage_occupancy_v<double, true, true, TY_DEFAULT>() : 1;
}
}  // namespace gbcfd
