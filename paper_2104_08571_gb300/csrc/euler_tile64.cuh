// FP64 2D first-order Euler steps, several per cooperative launch, sm_103a.
//
// What bounds it: the FP64 pipe.  Each of an SM's four schedulers issues one
// FP64 warp instruction in 64 clocks, so a warp alone keeps its scheduler's
// pipe busy, integer work and shared memory are free beside it, and the time
// of a step is the FP64 instructions of the most loaded scheduler.  So a
// tile's work is spread over whatever warps there are: primitive variables,
// physical fluxes and wave speeds once per cell of the tile and its halo, one
// face per lane, one update per lane, each list dealt out 32 items at a time
// to the warps in turn, with shared memory between the lists.  The tile's
// sides are chosen at run time so that the fullest scheduler has least to do.
//
// Per step, SoA, one launch a step on the tiles of euler_sweep.cuh (which form
// a state's primitives at each of its four faces) -> now: 64^2 17.5 -> 7.4 us,
// 128^2 17.4 -> 8.7 us, 512^2 104 -> 64 us, 1024^2 380 -> 240 us; AoS the same.
// (Strips walked by a warp, as the FP32 kernels have them, need three rows of
// primitives for a unit of one row: 14.1 us at 128^2, 257 us at 1024^2.)
#pragma once
#include "walk_common.cuh"

namespace ripple {

constexpr int kTile64Threads = 256;
constexpr int kTile64Cell = 12;  // doubles kept per cell: state 4, x flux 3, y flux 3, x and y speed
constexpr int kTile64Smem = 100 << 10;  // two CTAs per SM

// Bytes of shared memory of a tile of tx x ty cells.
__host__ __device__ constexpr int tile64_smem(int tx, int ty)
{
    return 8 * (kTile64Cell * (tx + 2) * (ty + 2) + 4 * ((tx + 1) * ty + tx * (ty + 1)));
}

__global__ void __launch_bounds__(kTile64Threads, 2) euler_tile64_kernel(const __grid_constant__ WalkStep a)
{
    extern __shared__ __align__(16) double tsm[];
    __shared__ double sdt[2];
    __shared__ double red[kTile64Threads / 32];
    __shared__ int sflag[1];
    const FieldGeom& g = a.g;
    FieldCtl* ctl = a.ctl;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nx = g.n[0], ny = g.n[1], tx = a.cols, ty = a.rows, pw = tx + 2;
    const int np = pw * (ty + 2), ncell = tx * ty, nhalo = ncell + 2 * (tx + ty);
    const int nxf = (tx + 1) * ty, nface = nxf + tx * (ty + 1);
    double* const fsm = tsm + kTile64Cell * np;  // faces: x faces [j][i], then y faces, component planes of nface
    const long long cs = g.comp_stride;
    const double gm1 = a.gamma - 1.0;
    const int tiles = a.strips * a.segs;
    if (tid == 0) sflag[0] = 0;
    for (int s = 0; s < a.K; ++s) {
        const int rs = (a.slot + s) % 3;
        const int cur = (a.cur + s) & 1;
        const double* __restrict__ in = reinterpret_cast<const double*>(a.buf[cur]);
        double* __restrict__ out = reinterpret_cast<double*>(a.buf[cur ^ 1]);
        double smax = 0.0;
        if (tid == kTile64Threads - 1) {
            // -dt / (2 dx) of each axis (faces carry a factor of two), once per CTA
            const double dt = a.cfl / __longlong_as_double((long long)__ldcg(&ctl->smax[rs]));
            sdt[0] = -0.5 * dt * a.inv_dx[0];
            sdt[1] = -0.5 * dt * a.inv_dx[1];
            if (blockIdx.x == 0) {
                ctl->t = s == 0 && a.first ? dt : ctl->t + dt;
                ctl->dt_last = dt;
                ctl->smax[(rs + 2) % 3] = 0ull;
            }
        }
        for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
            const int x0 = (tile % a.strips) * tx, y0 = (tile / a.strips) * ty;
            // cells of the tile, then of its four sides
            for (int e = tid; e < nhalo; e += kTile64Threads) {
                int i, j;
                if (e < ncell) {
                    j = e / tx;
                    i = e - j * tx;
                } else if (e < ncell + 2 * tx) {
                    const int k = e - ncell;
                    j = k < tx ? -1 : ty;
                    i = k < tx ? k : k - tx;
                } else {
                    const int k = e - ncell - 2 * tx;
                    i = k < ty ? -1 : tx;
                    j = k < ty ? k : k - ty;
                }
                const int x = x0 + i, y = y0 + j;
                // cells of the field and of its face ghosts (never a corner's)
                if (x > nx || y > ny || ((x < 0 || x == nx) && (y < 0 || y == ny))) continue;
                const double* p0 = in + geom_elem(g, x, y, 0, 0);
                double q[4];
#pragma unroll
                for (int m = 0; m < 4; ++m) q[m] = __ldcg(p0 + m * cs);
                const double ir = 1.0 / q[0];
                const double u = q[1] * ir, v = q[2] * ir;
                const double p = gm1 * (q[3] - 0.5 * fma(q[1], u, q[2] * v));
                const double c = sqrt(a.gamma * p * ir);
                const double h = q[3] + p;
                double* d = tsm + (j + 1) * pw + i + 1;
#pragma unroll
                for (int m = 0; m < 4; ++m) d[m * np] = q[m];
                d[4 * np] = fma(q[1], u, p);
                d[5 * np] = q[2] * u;
                d[6 * np] = h * u;
                d[7 * np] = q[1] * v;
                d[8 * np] = fma(q[2], v, p);
                d[9 * np] = h * v;
                d[10 * np] = fabs(u) + c;
                d[11 * np] = fabs(v) + c;
                if (!(q[0] > 0.0 && p > 0.0)) {
                    record_bad(ctl, BAD_STATE, x0, y0, 0);
                    atomicOr(&ctl->err, DEV_ERR_NUMERIC);
                }
            }
            __syncthreads();
            // twice the Rusanov flux of every face, x and y faces by the same code
            for (int e = tid; e < nface; e += kTile64Threads) {
                const bool fx = e < nxf;
                const int k = fx ? e : e - nxf, w = fx ? tx + 1 : tx;
                const int j = k / w, i = k - j * w;
                // cells beside the face: (i - 1, j) and (i, j), or (i, j - 1) and (i, j)
                if (x0 + i > (fx ? nx : nx - 1) || y0 + j > (fx ? ny - 1 : ny)) continue;
                const double* B = tsm + (j + 1) * pw + i + 1;
                const double* A = B - (fx ? 1 : pw);
                const int f1 = (fx ? 4 : 7) * np, sp = (fx ? 10 : 11) * np;
                const double sm = fmax(A[sp], B[sp]);
                const int f0 = (fx ? 1 : 2) * np;  // the mass flux is the momentum
                double* F = fsm + e;
                F[0] = fma(sm, A[0] - B[0], A[f0] + B[f0]);
#pragma unroll
                for (int m = 1; m < 4; ++m)
                    F[m * nface] = fma(sm, A[m * np] - B[m * np], A[f1 + (m - 1) * np] + B[f1 + (m - 1) * np]);
            }
            __syncthreads();
            const double kx = sdt[0], ky = sdt[1];
            for (int e = tid; e < ncell; e += kTile64Threads) {
                const int j = e / tx, i = e - j * tx;
                const int x = x0 + i, y = y0 + j;
                if (x >= nx || y >= ny) continue;
                const double* Q = tsm + (j + 1) * pw + i + 1;
                const double* Fx = fsm + j * (tx + 1) + i;
                const double* Fy = fsm + nxf + j * tx + i;
                double* po = out + geom_elem(g, x, y, 0, 0);
                double qn[4];
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const int o = m * nface;
                    qn[m] = fma(kx, Fx[o + 1] - Fx[o], fma(ky, Fy[o + tx] - Fy[o], Q[m * np]));
                    po[m * cs] = qn[m];
                }
                bool ok;
                smax = fmax(smax, wave_sum<double, 2>(qn, a.gamma, gm1, a.inv_dx, ok));
                if (!ok) {
                    record_bad(ctl, BAD_CELL, x, y, 0);
                    atomicOr(&ctl->err, DEV_ERR_NUMERIC);
                }
                if (x < g.h || x >= nx - g.h || y < g.h || y >= ny - g.h)
                    write_ghost_images<double, 2>(out, g, a.bc, x, y, 0, qn);
            }
            __syncthreads();
        }
        // CTA maximum of the new states' wave-speed sums into the next ring slot
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) smax = fmax(smax, __shfl_xor_sync(0xffffffffu, smax, o));
        if (lane == 0) red[warp] = smax;
        __syncthreads();
        if (tid == 0) {
            double m = red[0];
            for (int i = 1; i < kTile64Threads / 32; ++i) m = fmax(m, red[i]);
            atomic_max_pos_double(&ctl->smax[(rs + 1) % 3], m);
        }
        if (s + 1 < a.K && !grid_barrier(&ctl->bar[0], (unsigned)(s + 1), a.spin_limit, sflag)) break;
    }
    if (sflag[0] && tid == 0) atomicOr(a.err, DEV_ERR_TIMEOUT);
    walk_leave(ctl);
}

}  // namespace ripple
