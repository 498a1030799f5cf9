// Euler sweep kernels, element type double, 2D (all layouts, schemes, tiles),
// and the multi-step tiles of the first-order scheme.
#include "euler_tile64.cuh"
#include "sweep_table.cuh"

namespace ripple {
cudaError_t sweep_launch_f64_2d(int layout, int scheme, int v, const SweepLaunch& L)
{
    return SweepDim<double, 2>::launch(layout, scheme, v, L);
}
int sweep_smem_f64_2d(int layout, int scheme, int v) { return SweepDim<double, 2>::smem(layout, scheme, v); }
int sweep_occ_f64_2d(int layout, int scheme, int v) { return SweepDim<double, 2>::occ(layout, scheme, v); }
cudaError_t tile64_launch(const WalkStep& a, int grid, cudaStream_t s)
{
    void* args[] = {const_cast<WalkStep*>(&a)};
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(euler_tile64_kernel), dim3(grid),
                                       dim3(kTile64Threads), args, tile64_smem(a.cols, a.rows), s);
}
int tile64_occ()
{
    static ResidentCtas resident;
    return resident.get(euler_tile64_kernel, kTile64Threads, kTile64Smem);
}
// Sides of a tile: the ones that give the fullest SM the fewest FP64
// instructions per scheduler (counts per lane of the three lists of
// euler_tile64.cuh: 39, 13 and 51).  A tile alone on its SM takes whole rounds
// of four warps; tiles that follow one another fill each other's rounds, at a
// cost of about 16 instructions each for the CTA barriers.  Against the
// measured times per step (4 us + 0.033 us per instruction): 64^2 with 8 x 4
// tiles 7.4 us (modelled 7.4), 128^2 16 x 7 8.7 (9.1), 8 x 7 9.5 (9.7),
// 256^2 16 x 14 19.7 (20), 512^2 16 x 27 63.8 (64), 1024^2 16 x 27 240 (244),
// 32 x 17 258 (260), 16 x 7 270 (294).
void tile64_plan(WalkStep& a, int sms)
{
    const int nx = a.g.n[0], ny = a.g.n[1];
    double best = 1e300;
    for (int tx = 8; tx <= 32; tx *= 2)
        for (int ty = 1; ty <= 32 && tile64_smem(tx, ty) <= kTile64Smem; ++ty) {
            const long long ax = (nx + tx - 1) / tx, ay = (ny + ty - 1) / ty;
            // tiles of the fullest SM: one, or as many for each of its two CTAs
            const long long per = ax * ay <= sms ? 1 : 2 * ((ax * ay + 2 * sms - 1) / (2 * sms));
            auto rounds = [&](int items) {
                const int warps = (items + 31) / 32;
                return per > 1 ? 0.25 * warps : (double)((warps + 3) / 4);
            };
            const double cost = (double)per * (39 * rounds(tx * ty + 2 * (tx + ty)) + 51 * rounds(tx * ty) +
                                               13 * rounds((tx + 1) * ty + tx * (ty + 1)) + (per > 1 ? 16 : 0));
            if (cost < best) {
                best = cost;
                a.cols = tx;
                a.rows = ty;
                a.strips = (int)ax;
                a.segs = (int)ay;
            }
        }
}
}  // namespace ripple
