// FP32 2D and 3D steps of the dimensionally split FORCE solver (the paper's
// own Euler solver, Section 7.3, Listing euler_graph) on strip walks, sm_103a.
//
// One step is x, then y (then z) sweeps, each a flux difference along one
// axis of the state the sweep before it left.  The x and y sweeps are fused: a
// warp walks a strip of columns along y; each new row is swept along x in
// registers (neighbours and left faces by shuffles) and at once enters the y
// sweep as the upper row of a face, so the x-swept state never leaves the
// registers.  In 3D the walk stays in one z plane and writes the x- and
// y-swept state to the other buffer, and walks along z in a second phase of
// the same launch bring it back.  HBM traffic per cell update: 32 B in 2D (one
// sweep per launch moved 64 B), 80 B in 3D (120 B).
//
// Lanes: 64 columns x0 - 2 .. x0 + 61 of which the walk updates the 60 columns
// x0 .. x0 + 59; the two pairs at the ends only supply the x faces.  The pair
// width keeps every access of an aligned 8 bytes, and 60 of 64 costs less
// than a separate evaluation of the edge faces of every row.
// Rows: a walk updates rows y0 .. y1 - 1 and sweeps rows y0 - 1 .. y1 along x
// (two rows twice per segment).  A row outside the field is the interior row
// its ghost row would copy (walk_map): its x sweep gives the ghost row of the
// x-swept state, which is what refilling the padding between the sweeps gives.
// Faces shared by two walks are evaluated by both from the same values in the
// same order, so they have the same bits and the step stays conservative.
//
// The face: with a, b its states, F_a, F_b their physical fluxes (formed once
// per cell and handed to the neighbour), the flux of the Richtmyer state
//   q = (a + b)/2 - (dt/dx)/2 (F_b - F_a)
// is evaluated at 2q (the flux is homogeneous of degree one), and
//   V = F_a + F_b + F(2q) - (dx/dt)(b - a)
// is four times the FORCE flux; the factor goes into the update's dt/dx.
// Packed pair arithmetic throughout (pair_math.cuh).
//
// Staging: each lane copies its own pair of the coming rows into its part of
// a per-warp ring of kForceSlots slots with cp.async, so loads in flight hold
// no registers and no wait involves another thread.
//
// Measured (SoA, per step, one sweep per launch before -> now): 4096^2 250 ->
// 117 us, 256^3 630 -> 290 us, 200 x 171 x 186 300 -> 135 us, 64^3 19 us.
// Bound by issue: 164 thread instructions per cell update in 2D at 62 % issue;
// HBM would allow 80 us at 4096^2.
#pragma once
#include "walk_common.cuh"

namespace ripple {

constexpr int kForceSlots = 4;   // ring slots (rows) per warp
template <int DIM>
constexpr int force_smem() { return kWalkWarps * kForceSlots * 64 * (DIM + 2) * 4; }

// Four times the FORCE flux along D of the faces between a and b.
template <int DIM, int D>
__device__ __forceinline__ void force4(const f2 (&a)[DIM + 2], const f2 (&b)[DIM + 2], const f2 (&Fa)[DIM + 2],
                                       const f2 (&Fb)[DIM + 2], f2 gm1, f2 ndtdx, f2 ndxdt, f2 (&V)[DIM + 2])
{
    f2 q[DIM + 2], Fq[DIM + 2], iq, uq, pq;
#pragma unroll
    for (int m = 0; m < DIM + 2; ++m) q[m] = fma_v(ndtdx, Fb[m] - Fa[m], a[m] + b[m]);
    pflux<f2, DIM, D>(q, gm1, Fq, iq, uq, pq);
#pragma unroll
    for (int m = 0; m < DIM + 2; ++m) V[m] = fma_v(ndxdt, b[m] - a[m], (Fa[m] + Fb[m]) + Fq[m]);
}

struct ForceConsts {
    f2 gamma, gm1, ivx[3];
    f2 ndtdx[3], ndxdt[3], nc[3];  // -dt/dx, -dx/dt, -(dt/dx)/4
};

// One walk: rows r0 .. r1 - 1 along axis D (1: y, 2: z) of the pair columns
// starting at x0; XS: sweep every row along x first; LAST: the step's last
// sweep (wave speeds, admissibility and ghost images of the new state).
// `line` is the z plane of a y walk, the y row of a z walk.  begin() stages
// the walk's first rows, which needs no dt; run() walks.
template <int DIM, int LAYOUT, int D, bool XS, bool LAST>
struct ForceWalk {
    static constexpr int NC = DIM + 2, NS = kForceSlots, SLOT = 64 * NC;
    static constexpr long long CST = LAYOUT == LAYOUT_SOA ? 1 : NC;
    WalkRows rows;
    int x0, r0, r1, line;
    long long org, stride;

    __device__ __forceinline__ void begin(const float* __restrict__ in, const WalkStep& a, int x0_, int r0_, int r1_,
                                          int line_, float* ring, int lane)
    {
        const FieldGeom& g = a.g;
        x0 = x0_; r0 = r0_; r1 = r1_; line = line_;
        stride = (D == 1 ? g.px : g.px * g.py) * CST;
        // element offset of x = 0 in row 0 (pairs past the field read the last pair that holds a ghost cell)
        const long long zoff = DIM == 3 ? (long long)(g.h + (D == 1 ? line : 0)) * g.py : 0;
        org = ((zoff + g.h + (D == 1 ? 0 : line)) * g.px + g.lead + g.h) * CST;
        rows.init(in + org + min(x0 + 2 * lane, g.n[0] & ~1) * CST, stride, r0 - 1, g.n[D], a.bc);
        const int n = r1 - r0 + 2;
#pragma unroll
        for (int i = 0; i < NS - 1; ++i) {
            if (i < n) {
                walk_stage<DIM, LAYOUT>(ring + i * SLOT, lane, rows.p, g.comp_stride);
                rows.next();
            }
            cp_async_commit();
        }
    }

    __device__ __forceinline__ void run(float* __restrict__ out, const WalkStep& a, float* ring, int lane,
                                        const ForceConsts& k, float& smax);
};

template <int DIM, int LAYOUT, int D, bool XS, bool LAST>
__device__ __forceinline__ void ForceWalk<DIM, LAYOUT, D, XS, LAST>::run(float* __restrict__ out, const WalkStep& a,
                                                                        float* ring, int lane, const ForceConsts& k,
                                                                        float& smax)
{
    const FieldGeom& g = a.g;
    const int nx = g.n[0], na = g.n[D];
    const int x = x0 + 2 * lane;
    const bool v0 = (!XS || (lane >= 1 && lane <= 30)) && x < nx, v1 = v0 && x + 1 < nx;
    const long long cs = g.comp_stride;
    float* const po0 = out + org + x * CST + r0 * stride;
    float* po = po0;
    const int n = r1 - r0 + 2;
    float cx = 1.f, c0 = 1.f, c1 = 1.f;  // smallest density/pressure: before the x sweep, after it (per cell)
    WalkNew nw;
    const bool full = x0 + 64 <= nx;  // every pair that is updated lies in the field
    const bool edge_x = LAST && (x0 < g.h || x0 + 64 > nx - g.h);
    const int nl = DIM == 3 ? g.n[D == 1 ? 2 : 1] : 1;  // lines across the walk's plane
    const bool edge_l = LAST && DIM == 3 && (line < g.h || line >= nl - g.h);
    float* rd = ring;                      // slot of row i
    float* wr = ring + (NS - 1) * SLOT;    // slot of row i + NS - 1
    // row i = 0 .. n - 1 of the walk (r0 - 1 + i) from the row before it: `a` holds
    // the swept row, its flux along D and the face below it, `b` receives this row's
    auto row = [&](int i, const f2 (&qa)[NC], const f2 (&Fa)[NC], const f2 (&Va)[NC], f2 (&qb)[NC], f2 (&Fb)[NC],
                   f2 (&Vb)[NC]) {
        if (i + NS - 1 < n) {
            walk_stage<DIM, LAYOUT>(wr, lane, rows.p, cs);
            rows.next();
        }
        cp_async_commit();
        cp_async_wait<NS - 1>();
        f2 ir, un, p;
        if constexpr (XS) {
            f2 q[NC], F[NC], b[NC], G[NC], V[NC];
            walk_read<DIM, LAYOUT>(rd, lane, q);
            pflux<f2, DIM, 0>(q, k.gm1, F, ir, un, p);
            cx = min3f(cx, q[0].x, p.x);
            cx = min3f(cx, q[0].y, p.y);
#pragma unroll
            for (int m = 0; m < NC; ++m) b[m] = f2{q[m].y, __shfl_down_sync(0xffffffffu, q[m].x, 1)};
            G[0] = b[1];
#pragma unroll
            for (int m = 1; m < NC; ++m) G[m] = f2{F[m].y, __shfl_down_sync(0xffffffffu, F[m].x, 1)};
            force4<DIM, 0>(q, b, F, G, k.gm1, k.ndtdx[0], k.ndxdt[0], V);
#pragma unroll
            for (int m = 0; m < NC; ++m) {
                const f2 Vl = f2{__shfl_up_sync(0xffffffffu, V[m].y, 1), V[m].x};
                qb[m] = fma_v(k.nc[0], V[m] - Vl, q[m]);
            }
        } else {
            walk_read<DIM, LAYOUT>(rd, lane, qb);
        }
        pflux<f2, DIM, D>(qb, k.gm1, Fb, ir, un, p);
        c0 = min3f(c0, qb[0].x, p.x);
        c1 = min3f(c1, qb[0].y, p.y);
        force4<DIM, D>(qa, qb, Fa, Fb, k.gm1, k.ndtdx[D], k.ndxdt[D], Vb);
        if (i >= 2) {
            f2 qn[NC];
#pragma unroll
            for (int m = 0; m < NC; ++m) qn[m] = fma_v(k.nc[D], Vb[m] - Va[m], qa[m]);
            walk_store<DIM, LAYOUT>(po, cs, qn, v0, v1, full);
            if constexpr (LAST) {
                const int r = r0 + i - 2;
                if (edge_x) walk_ghost_x<DIM, LAYOUT>(po, cs, qn, x, nx, g.h, a.bc, v0, v1);
                if (r < g.h || r >= na - g.h)
                    walk_ghost_rows<DIM, LAYOUT>(po, cs, qn, r, na, g.h, a.bc, stride, v0, v1, full);
                if (edge_l)
                    walk_ghost_rows<DIM, LAYOUT>(po, cs, qn, line, nl, g.h, a.bc, (D == 1 ? g.px * g.py : g.px) * CST,
                                                 v0, v1, full);
                nw.add<DIM>(qn, k.gamma, k.gm1, k.ivx);
            }
            po += stride;
        }
        __syncwarp();  // the lanes part at the field's edges: bring them together once a row
        wr = rd;
        rd = rd == ring + (NS - 1) * SLOT ? ring : rd + SLOT;
    };
    f2 q0[NC], F0[NC], V0[NC], q1[NC], F1[NC], V1[NC];
#pragma unroll
    for (int m = 0; m < NC; ++m) q0[m] = F0[m] = V0[m] = f2{1.f, 1.f};  // the first face of a walk is not used
    // two rows per iteration, so that what passes from row to row changes hands without copies
#pragma unroll 1
    for (int i = 0; i < n; i += 2) {
        row(i, q0, F0, V0, q1, F1, V1);
        if (i + 1 >= n) break;
        row(i + 1, q1, F1, V1, q0, F0, V0);
    }
    if constexpr (LAST) smax = fmaxf(smax, fmaxf(v0 ? nw.s0 : 0.f, v1 ? nw.s1 : 0.f));
    // a non-admissible state on some face of the walk (columns outside the
    // walk or the field are copies, padding (NaN) or undefined after the sweep)
    if ((XS && !(cx > 0.f)) || (v0 && !(c0 > 0.f)) || (v1 && !(c1 > 0.f))) {
        record_bad(a.ctl, BAD_STATE, max(x, 0), D == 1 ? r0 : line, D == 1 ? line : r0);
        atomicOr(&a.ctl->err, DEV_ERR_NUMERIC);
    }
    if constexpr (LAST) {
        const long long cstr = LAYOUT == LAYOUT_SOA ? cs : 1;
        if (v0 && !nw.ok0) walk_bad_cell<DIM>(a.ctl, a.gamma_f, a.gm1_f, po0, stride, cstr, D, x, line, r0, r1);
        if (v1 && !nw.ok1) walk_bad_cell<DIM>(a.ctl, a.gamma_f, a.gm1_f, po0 + CST, stride, cstr, D, x + 1, line, r0, r1);
    }
}

template <int DIM, int LAYOUT>
__global__ void __launch_bounds__(kWalkWarps * 32, 1) euler_force_walk_kernel(const __grid_constant__ WalkStep a)
{
    constexpr int NC = DIM + 2;
    extern __shared__ __align__(128) float wsm[];
    __shared__ float sdt[9];
    __shared__ float red[kWalkWarps];
    __shared__ int sflag[1];
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    float* ring = wsm + warp * kForceSlots * 64 * NC;
    FieldCtl* ctl = a.ctl;
    ForceConsts k;
    k.gamma = splat<f2>(a.gamma_f);
    k.gm1 = splat<f2>(a.gm1_f);
#pragma unroll
    for (int d = 0; d < 3; ++d) k.ivx[d] = splat<f2>(a.inv_dx_f[d]);
    if (tid == 0) sflag[0] = 0;
    unsigned phase = 0;  // a barrier ends every phase but the last
    for (int s = 0; s < a.K; ++s) {
        const int rs = (a.slot + s) % 3;
        const int cur = DIM == 3 ? a.cur : (a.cur + s) & 1;
        float* A = a.buf[cur];
        float* B = a.buf[cur ^ 1];
        ForceWalk<DIM, LAYOUT, 1, true, DIM == 2> w;
        const int per = a.strips * a.segs;
        WalkUnits todo(ctl, phase, DIM == 3 ? per * a.g.n[2] : per, lane, warp);
        auto begin = [&]() {
            if (!todo.any()) return;
            const int pl = DIM == 3 ? todo.u / per : 0, v = DIM == 3 ? todo.u % per : todo.u;
            const int strip = v % a.strips, r0 = (v / a.strips) * a.rows;
            w.begin(A, a, strip * kWalkUse - 2, r0, min(a.g.n[1], r0 + a.rows), pl, ring, lane);
        };
        begin();
        if (tid == 0) {
            // dt from the largest wave-speed sum of the step's input state, in FP64 once per CTA
            const double sm = __longlong_as_double((long long)__ldcg(&ctl->smax[rs]));
            const double dt = a.cfl / sm;
            for (int d = 0; d < DIM; ++d) {
                sdt[d] = (float)(-dt * a.inv_dx[d]);
                sdt[3 + d] = (float)(-sm * a.dx_cfl[d]);
                sdt[6 + d] = (float)(-0.25 * dt * a.inv_dx[d]);
            }
            if (blockIdx.x == 0) {
                ctl->t = s == 0 && a.first ? dt : ctl->t + dt;
                ctl->dt_last = dt;
                ctl->smax[(rs + 2) % 3] = 0ull;
            }
        }
        __syncthreads();
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            k.ndtdx[d] = splat<f2>(sdt[d]);
            k.ndxdt[d] = splat<f2>(sdt[3 + d]);
            k.nc[d] = splat<f2>(sdt[6 + d]);
        }
        float smax = 0.f;
        while (todo.any()) {
            todo.ask();
            w.run(B, a, ring, lane, k, smax);
            todo.advance();
            begin();
        }
        if constexpr (DIM == 3) {
            if (!grid_barrier(&ctl->bar[0], ++phase, a.spin_limit, sflag)) break;
            const int zper = a.zstrips * a.g.n[1];
            ForceWalk<DIM, LAYOUT, DIM - 1, false, true> wz;
            for (WalkUnits zt(ctl, phase, zper * a.zsegs, lane, warp); zt.any(); zt.advance()) {
                zt.ask();
                const int v = zt.u % zper, r0 = (zt.u / zper) * a.zrows;
                wz.begin(B, a, (v % a.zstrips) * 64, r0, min(a.g.n[2], r0 + a.zrows), v / a.zstrips, ring, lane);
                wz.run(A, a, ring, lane, k, smax);
            }
        }
        walk_reduce(ctl, (rs + 1) % 3, smax, red);
        if (s + 1 < a.K && !grid_barrier(&ctl->bar[0], ++phase, a.spin_limit, sflag)) break;
    }
    if (sflag[0] && tid == 0) atomicOr(a.err, DEV_ERR_TIMEOUT);
    walk_leave(ctl);
}

}  // namespace ripple

#include "resident.h"
#include "runtime.h"

namespace ripple {

template <int DIM, int LAYOUT>
static int force_walk_occupancy()  // resident CTAs per SM, 0 if the kernel cannot run
{
    static ResidentCtas resident;
    return resident.get(euler_force_walk_kernel<DIM, LAYOUT>, kWalkWarps * 32, force_smem<DIM>());
}
template <int DIM, int LAYOUT>
static cudaError_t force_walk_run(const WalkStep& a, int grid, cudaStream_t s)
{
    void* args[] = {const_cast<WalkStep*>(&a)};
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(euler_force_walk_kernel<DIM, LAYOUT>), dim3(grid),
                                       dim3(kWalkWarps * 32), args, force_smem<DIM>(), s);
}

}  // namespace ripple
