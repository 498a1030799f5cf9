// Euler sweep kernels, element type float, 2D (all layouts, schemes, tiles),
// and the strip walks of the split FORCE step.
#include "euler_force_walk.cuh"
#include "euler_walk2d.cuh"
#include "sweep_table.cuh"

namespace ripple {
cudaError_t sweep_launch_f32_2d(int layout, int scheme, int v, const SweepLaunch& L)
{
    return SweepDim<float, 2>::launch(layout, scheme, v, L);
}
int sweep_smem_f32_2d(int layout, int scheme, int v) { return SweepDim<float, 2>::smem(layout, scheme, v); }
int sweep_occ_f32_2d(int layout, int scheme, int v) { return SweepDim<float, 2>::occ(layout, scheme, v); }

cudaError_t force_walk_launch_f32_2d(int layout, const WalkStep& a, int grid, cudaStream_t s)
{
    return layout == LAYOUT_SOA ? force_walk_run<2, LAYOUT_SOA>(a, grid, s) : force_walk_run<2, LAYOUT_AOS>(a, grid, s);
}
int force_walk_occ_f32_2d(int layout)
{
    return layout == LAYOUT_SOA ? force_walk_occupancy<2, LAYOUT_SOA>() : force_walk_occupancy<2, LAYOUT_AOS>();
}

cudaError_t walk2d_launch_f32(int scheme, int layout, const WalkStep& a, int grid, cudaStream_t s)
{
    if (scheme == SCHEME_MUSCL)
        return layout == LAYOUT_SOA ? walk2d_run<SCHEME_MUSCL, LAYOUT_SOA>(a, grid, s)
                                    : walk2d_run<SCHEME_MUSCL, LAYOUT_AOS>(a, grid, s);
    return layout == LAYOUT_SOA ? walk2d_run<SCHEME_RUSANOV1, LAYOUT_SOA>(a, grid, s)
                                : walk2d_run<SCHEME_RUSANOV1, LAYOUT_AOS>(a, grid, s);
}
int walk2d_occ_f32(int scheme, int layout)
{
    if (scheme == SCHEME_MUSCL)
        return layout == LAYOUT_SOA ? walk2d_occupancy<SCHEME_MUSCL, LAYOUT_SOA>()
                                    : walk2d_occupancy<SCHEME_MUSCL, LAYOUT_AOS>();
    return layout == LAYOUT_SOA ? walk2d_occupancy<SCHEME_RUSANOV1, LAYOUT_SOA>()
                                : walk2d_occupancy<SCHEME_RUSANOV1, LAYOUT_AOS>();
}
}  // namespace ripple
