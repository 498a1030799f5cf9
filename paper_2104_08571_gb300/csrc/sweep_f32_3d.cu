// Euler sweep kernels, element type float, 3D (all layouts, schemes, tiles),
// and the strip walks of the split FORCE step.
#include "euler_force_walk.cuh"
#include "sweep_table.cuh"

namespace ripple {
cudaError_t sweep_launch_f32_3d(int layout, int scheme, int v, const SweepLaunch& L)
{
    return SweepDim<float, 3>::launch(layout, scheme, v, L);
}
int sweep_smem_f32_3d(int layout, int scheme, int v) { return SweepDim<float, 3>::smem(layout, scheme, v); }
int sweep_occ_f32_3d(int layout, int scheme, int v) { return SweepDim<float, 3>::occ(layout, scheme, v); }

cudaError_t force_walk_launch_f32_3d(int layout, const WalkStep& a, int grid, cudaStream_t s)
{
    return layout == LAYOUT_SOA ? force_walk_run<3, LAYOUT_SOA>(a, grid, s) : force_walk_run<3, LAYOUT_AOS>(a, grid, s);
}
int force_walk_occ_f32_3d(int layout)
{
    return layout == LAYOUT_SOA ? force_walk_occupancy<3, LAYOUT_SOA>() : force_walk_occupancy<3, LAYOUT_AOS>();
}
}  // namespace ripple
