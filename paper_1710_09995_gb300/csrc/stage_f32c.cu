// stage_f32c.cu -- stage-kernel instantiations: mixed path (f32 fluxes), curvilinear grids
#include "stage_c.cuh"

namespace gbcfd {
cudaError_t launch_stage_f32c(int viscous, int stage, const GroupParams& P, int grid,
                              cudaStream_t s) {
  return viscous ? cstage_dispatch<true, TY_DEFAULT>(stage, P, grid, s)
                 : cstage_dispatch<false, TY_DEFAULT>(stage, P, grid, s);
}
cudaError_t stage_prepare_f32c(int viscous) {
  return viscous ? cstage_prepare<true, TY_DEFAULT>() : cstage_prepare<false, TY_DEFAULT>();
}
int stage_occupancy_f32c(int) { return 1; }  // the metric ring takes the SM
}  // namespace gbcfd
