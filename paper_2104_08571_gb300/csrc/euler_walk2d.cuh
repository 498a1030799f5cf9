// FP32 2D unsplit Euler steps (first-order Rusanov, MUSCL-Hancock) on strip
// walks, sm_103a.
//
// One cooperative launch advances the field K steps; a step is one pass of
// all warps over their walks and a grid barrier (walk_common.cuh).  A warp
// walks rows y0 .. y1 - 1 of the 60 columns x0 .. x0 + 59 (lanes hold
// x0 - 2 .. x0 + 61 as pairs: two halo columns on either side, which is what
// MUSCL-Hancock needs and what keeps every pair 8-byte aligned).  Along x a
// cell's neighbours and its left face come from the next lanes by shuffles;
// along y the predicted high state and the face below a row stay in registers
// from row to row, and the row's x flux difference waits one row for the face
// above it.  Every face and predicted state of a walk is formed once; a
// segment adds two rows of predicted states and one of faces.
//
// What bounds it: instruction issue.  The tiles of euler_sweep_pair.cuh pass
// predicted states and faces through shared memory between three CTA barriers
// a tile; the walk has none of those, and small grids also save the launch of
// every step.  Measured per step (SoA, tiles before -> now): MUSCL-Hancock
// 1000 x 701 27.8 -> 13.7 us, 64^2 8.3 -> 4.8 us; Rusanov 64^2 8.3 -> 4.0 us,
// 1024^2 22.6 -> 11.2 us.
#pragma once
#include "walk_common.cuh"

namespace ripple {

template <int SCHEME>
struct Walk2D {
    static constexpr bool MH = SCHEME == SCHEME_MUSCL;
    static constexpr int SLOTS = MH ? 6 : 4;  // ring rows per warp: the rows of a stencil and two or three ahead
    static constexpr int SMEM = kWalkWarps * SLOTS * 64 * 4 * 4;
};

struct Walk2DConsts {
    f2 gamma, gm1, ivx[3];
    f2 hdtdx[2];  // (dt/dx)/2 (predictor)
    f2 mdt;       // -dt
};

// Twice the Rusanov flux between a and b from their physical fluxes and wave
// speeds |u| + c.
__device__ __forceinline__ void rus2_pre(const f2 (&a)[4], const f2 (&b)[4], const f2 (&Fa)[4], const f2 (&Fb)[4],
                                         f2 sa, f2 sb, f2 (&V)[4])
{
    const f2 s = max_v(sa, sb);
#pragma unroll
    for (int m = 0; m < 4; ++m) V[m] = fma_v(s, a[m] - b[m], Fa[m] + Fb[m]);
}

// One walk: rows r0 .. r1 - 1 of the strip whose lanes start at column x0.
// begin() stages the walk's first rows, which needs no dt; run() walks.  `a`
// describes the problem (g, bc, ctl, gamma_f, gm1_f): a WalkStep, or an
// instance of the batched step.
template <int SCHEME, int LAYOUT>
struct PlaneWalk {
    static constexpr bool MH = SCHEME == SCHEME_MUSCL;
    static constexpr int NC = 4, NS = Walk2D<SCHEME>::SLOTS, SLOT = 64 * NC;
    static constexpr int R = MH ? 2 : 1, W = MH ? 3 : 1;  // stencil radius, rows read per iteration
    static constexpr long long CST = LAYOUT == LAYOUT_SOA ? 1 : NC;
    WalkRows rows;
    int x0, r0, r1;

    template <class A>
    __device__ __forceinline__ void begin(const float* __restrict__ in, const A& a, int x0_, int r0_, int r1_,
                                          float* ring, int lane)
    {
        const FieldGeom& g = a.g;
        x0 = x0_; r0 = r0_; r1 = r1_;
        const long long org = (g.h * g.px + g.lead + g.h) * CST;
        // pairs past the field read the last pair that holds a ghost cell (MUSCL-Hancock: ghost nx + 1)
        rows.init(in + org + min(x0 + 2 * lane, (MH ? g.n[0] + 1 : g.n[0]) & ~1) * CST, g.px * CST, r0 - R, g.n[1],
                  a.bc);
        const int nr = r1 - r0 + 2 * R;  // rows read: r0 - R .. r1 + R - 1
#pragma unroll
        for (int j = 0; j < NS - 1; ++j) {
            if (j < nr) {
                walk_stage<2, LAYOUT>(ring + j * SLOT, lane, rows.p, g.comp_stride);
                rows.next();
            }
            cp_async_commit();
        }
    }

    template <class A>
    __device__ __forceinline__ void run(float* __restrict__ out, const A& a, float* ring, int lane,
                                        const Walk2DConsts& k, float& smax);
};

template <int SCHEME, int LAYOUT>
template <class A>
__device__ __forceinline__ void PlaneWalk<SCHEME, LAYOUT>::run(float* __restrict__ out, const A& a, float* ring,
                                                               int lane, const Walk2DConsts& k, float& smax)
{
    const FieldGeom& g = a.g;
    const int nx = g.n[0], ny = g.n[1];
    const int x = x0 + 2 * lane;
    const bool v0 = lane >= 1 && lane <= 30 && x < nx, v1 = v0 && x + 1 < nx;
    const long long cs = g.comp_stride, stride = g.px * CST;
    float* const po0 = out + (g.h * g.px + g.lead + g.h) * CST + x * CST + r0 * stride;
    float* po = po0;
    const int n = r1 - r0 + 2;  // rows r0 - 1 .. r1
    const int nr = n + W - 1;   // rows read
    f2 cx = f2{1.f, 1.f}, cy = f2{1.f, 1.f};  // smallest density/pressure of the states on x and y faces, per column
    WalkNew nw;
    const bool full = x0 + 64 <= nx;
    const bool edge_x = x0 < g.h || x0 + 64 > nx - g.h;
    float* const last = ring + (NS - 1) * SLOT;
    float* rd = ring;  // slot of the first row read in this iteration
    float* wr = last;  // slot of the row staged in this iteration
    // row r0 - 1 + i from the row before it: `a` holds of that row the high y
    // state (MH) or the state, its y flux and speed (first order), the face below
    // it and its x part; `b` receives this row's
    auto row = [&](int i, const f2 (&Ya)[NC], const f2 (&Va)[NC], const f2 (&Xa)[NC], const f2 (&qa)[NC], const f2& sa,
                   f2 (&Yb)[NC], f2 (&Vb)[NC], f2 (&Xb)[NC], f2 (&qb)[NC], f2& sb) {
        if (i + NS - 1 < nr) {
            walk_stage<2, LAYOUT>(wr, lane, rows.p, cs);
            rows.next();
        }
        cp_async_commit();
        cp_async_wait<NS - W>();  // rows i .. i + W - 1 of the walk have landed
        const bool inner = i >= 1 && i <= n - 2;
        f2 q[NC], qm[NC];
        if constexpr (MH) {
            f2 L[NC], H[NC];
            {
                f2 qq[NC];
                const float* s1 = rd == last ? ring : rd + SLOT;
                const float* s2 = s1 == last ? ring : s1 + SLOT;
                walk_read<2, LAYOUT>(rd, lane, qm);
                walk_read<2, LAYOUT>(s1, lane, q);
                walk_read<2, LAYOUT>(s2, lane, qq);
                muscl<f2, 2, 1>(qm, q, qq, k.gm1, k.hdtdx[1], L, Yb, cy);
            }
            rus2<2, 1>(Ya, L, k.gamma, k.gm1, Vb, cy);
            if (inner) {
                f2 ql[NC], qr[NC], F[NC];
#pragma unroll
                for (int m = 0; m < NC; ++m) {
                    ql[m] = f2{__shfl_up_sync(0xffffffffu, q[m].y, 1), q[m].x};
                    qr[m] = f2{q[m].y, __shfl_down_sync(0xffffffffu, q[m].x, 1)};
                }
                muscl<f2, 2, 0>(ql, q, qr, k.gm1, k.hdtdx[0], L, H, cx);
#pragma unroll
                for (int m = 0; m < NC; ++m) qr[m] = f2{L[m].y, __shfl_down_sync(0xffffffffu, L[m].x, 1)};
                rus2<2, 0>(H, qr, k.gamma, k.gm1, F, cx);
#pragma unroll
                for (int m = 0; m < NC; ++m) Xb[m] = F[m] - f2{__shfl_up_sync(0xffffffffu, F[m].y, 1), F[m].x};
            }
        } else {
            walk_read<2, LAYOUT>(rd, lane, qb);
            f2 Fx[NC], ir, u, v, p;
            pflux<f2, 2, 0>(qb, k.gm1, Fx, ir, u, p);
            cx.x = min3f(cx.x, qb[0].x, p.x);
            cx.y = min3f(cx.y, qb[0].y, p.y);
            const f2 c = sqrt_v(k.gamma * p * ir);
            const f2 sx = abs_v(u) + c;
            pflux_y(qb, ir, p, Yb, v);
            sb = abs_v(v) + c;
            rus2_pre(qa, qb, Ya, Yb, sa, sb, Vb);
            if (inner) {
                f2 b[NC], Fb[NC], F[NC];
#pragma unroll
                for (int m = 0; m < NC; ++m) b[m] = f2{qb[m].y, __shfl_down_sync(0xffffffffu, qb[m].x, 1)};
                Fb[0] = b[1];
#pragma unroll
                for (int m = 1; m < NC; ++m) Fb[m] = f2{Fx[m].y, __shfl_down_sync(0xffffffffu, Fx[m].x, 1)};
                rus2_pre(qb, b, Fx, Fb, sx, f2{sx.y, __shfl_down_sync(0xffffffffu, sx.x, 1)}, F);
#pragma unroll
                for (int m = 0; m < NC; ++m) Xb[m] = F[m] - f2{__shfl_up_sync(0xffffffffu, F[m].y, 1), F[m].x};
            }
        }
        if (i >= 2) {
            // update of row r - 1 = r0 + i - 2 (faces carry a factor of two)
            const int r = r0 + i - 2;
            f2 qn[NC];
#pragma unroll
            for (int m = 0; m < NC; ++m)
                qn[m] = fma_v(k.mdt, fma_v(Vb[m] - Va[m], k.ivx[1], Xa[m] * k.ivx[0]), MH ? qm[m] : qa[m]);
            walk_store<2, LAYOUT>(po, cs, qn, v0, v1, full);
            if (edge_x) walk_ghost_x<2, LAYOUT>(po, cs, qn, x, nx, g.h, a.bc, v0, v1);
            if (r < g.h || r >= ny - g.h)
                walk_ghost_rows<2, LAYOUT>(po, cs, qn, r, ny, g.h, a.bc, stride, v0, v1, full);
            po += stride;
            nw.add<2>(qn, k.gamma, k.gm1, k.ivx);
        }
        __syncwarp();  // the lanes part at the field's edges: bring them together once a row
        wr = rd;
        rd = rd == last ? ring : rd + SLOT;
    };
    f2 Y0[NC], V0[NC], X0[NC], q0[NC], s0, Y1[NC], V1[NC], X1[NC], q1[NC], s1;
#pragma unroll
    for (int m = 0; m < NC; ++m) {
        // the first face of a walk is not used; its lower state is admissible (density 1, at rest)
        Y0[m] = q0[m] = m == 0 || m == NC - 1 ? f2{1.f, 1.f} : f2{0.f, 0.f};
        V0[m] = X0[m] = X1[m] = f2{0.f, 0.f};
    }
    s0 = f2{0.f, 0.f};
    // two rows per iteration, so that what passes from row to row changes hands without copies
#pragma unroll 1
    for (int i = 0; i < n; i += 2) {
        row(i, Y0, V0, X0, q0, s0, Y1, V1, X1, q1, s1);
        if (i + 1 >= n) break;
        row(i + 1, Y1, V1, X1, q1, s1, Y0, V0, X0, q0, s0);
    }
    smax = fmaxf(smax, fmaxf(v0 ? nw.s0 : 0.f, v1 ? nw.s1 : 0.f));
    // non-admissible states on the walk's faces: x faces of the columns -1 .. nx
    // (first order: every state read is a cell's or its ghost's), y faces of its own
    const bool bx = MH ? (x + 1 <= nx && !(cx.x > 0.f)) || (x + 2 <= nx && lane < 31 && !(cx.y > 0.f))
                       : !(cx.x > 0.f) || !(cx.y > 0.f);
    if (bx || (v0 && !(cy.x > 0.f)) || (v1 && !(cy.y > 0.f))) {
        record_bad(a.ctl, BAD_STATE, max(x, 0), r0, 0);
        atomicOr(&a.ctl->err, DEV_ERR_NUMERIC);
    }
    const long long cstr = LAYOUT == LAYOUT_SOA ? cs : 1;
    if (v0 && !nw.ok0) walk_bad_cell<2>(a.ctl, a.gamma_f, a.gm1_f, po0, stride, cstr, 1, x, 0, r0, r1);
    if (v1 && !nw.ok1) walk_bad_cell<2>(a.ctl, a.gamma_f, a.gm1_f, po0 + CST, stride, cstr, 1, x + 1, 0, r0, r1);
}

template <int SCHEME, int LAYOUT>
__global__ void __launch_bounds__(kWalkWarps * 32, 1) euler_walk2d_kernel(const __grid_constant__ WalkStep a)
{
    extern __shared__ __align__(128) float wsm[];
    __shared__ float sdt[3];
    __shared__ float red[kWalkWarps];
    __shared__ int sflag[1];
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    float* ring = wsm + warp * Walk2D<SCHEME>::SLOTS * 64 * 4;
    FieldCtl* ctl = a.ctl;
    Walk2DConsts k;
    k.gamma = splat<f2>(a.gamma_f);
    k.gm1 = splat<f2>(a.gm1_f);
#pragma unroll
    for (int d = 0; d < 3; ++d) k.ivx[d] = splat<f2>(a.inv_dx_f[d]);
    if (tid == 0) sflag[0] = 0;
    for (int s = 0; s < a.K; ++s) {
        const int rs = (a.slot + s) % 3;
        const int cur = (a.cur + s) & 1;
        PlaneWalk<SCHEME, LAYOUT> w;
        WalkUnits todo(ctl, (unsigned)s, a.strips * a.segs, lane, warp);
        auto begin = [&]() {
            if (!todo.any()) return;
            const int r0 = (todo.u / a.strips) * a.rows;
            w.begin(a.buf[cur], a, (todo.u % a.strips) * kWalkUse - 2, r0, min(a.g.n[1], r0 + a.rows), ring, lane);
        };
        begin();
        if (tid == 0) {
            // dt from the largest wave-speed sum of the step's input state, in FP64 once per CTA
            const double dt = a.cfl / __longlong_as_double((long long)__ldcg(&ctl->smax[rs]));
            sdt[0] = (float)(-0.5 * dt);
            for (int d = 0; d < 2; ++d) sdt[1 + d] = (float)(0.5 * dt * a.inv_dx[d]);
            if (blockIdx.x == 0) {
                ctl->t = s == 0 && a.first ? dt : ctl->t + dt;
                ctl->dt_last = dt;
                ctl->smax[(rs + 2) % 3] = 0ull;
            }
        }
        __syncthreads();
        k.mdt = splat<f2>(sdt[0]);
        k.hdtdx[0] = splat<f2>(sdt[1]);
        k.hdtdx[1] = splat<f2>(sdt[2]);
        float smax = 0.f;
        while (todo.any()) {
            todo.ask();
            w.run(a.buf[cur ^ 1], a, ring, lane, k, smax);
            todo.advance();
            begin();
        }
        walk_reduce(ctl, (rs + 1) % 3, smax, red);
        if (s + 1 < a.K && !grid_barrier(&ctl->bar[0], (unsigned)(s + 1), a.spin_limit, sflag)) break;
    }
    if (sflag[0] && tid == 0) atomicOr(a.err, DEV_ERR_TIMEOUT);
    walk_leave(ctl);
}

}  // namespace ripple

#include "resident.h"
#include "runtime.h"

namespace ripple {

template <int SCHEME, int LAYOUT>
static int walk2d_occupancy()
{
    static ResidentCtas resident;
    return resident.get(euler_walk2d_kernel<SCHEME, LAYOUT>, kWalkWarps * 32, Walk2D<SCHEME>::SMEM);
}
template <int SCHEME, int LAYOUT>
static cudaError_t walk2d_run(const WalkStep& a, int grid, cudaStream_t s)
{
    void* args[] = {const_cast<WalkStep*>(&a)};
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(euler_walk2d_kernel<SCHEME, LAYOUT>), dim3(grid),
                                       dim3(kWalkWarps * 32), args, Walk2D<SCHEME>::SMEM, s);
}

}  // namespace ripple
