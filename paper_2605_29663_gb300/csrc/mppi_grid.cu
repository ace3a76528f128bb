// mppi_grid.cu -- the control cycles (static clouds, and clouds with point
// velocities) whose sample phase walks the cloud's cell grid; see
// cloud_grid.cuh.  Only the instantiations live here, so they compile in
// parallel with mppi.cu.
#include "mppi_kernels.cuh"

namespace exact {

// V.vel: one grid for a cloud whose points move (see kStepGridBytes); a cloud
// with a grid per step is walked like a static one.
int launch_cycle_grid(const SceneView &V, const exact_footprint *fp, cudaStream_t st, const CloudGrid *grid,
                      GridStride gst, int sms) {
    return V.vel ? launch_grid_cycle_t<true>(V, fp, st, grid, gst, sms)
                 : launch_grid_cycle_t<false>(V, fp, st, grid, gst, sms);
}

}  // namespace exact
