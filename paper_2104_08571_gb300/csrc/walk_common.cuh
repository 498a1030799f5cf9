// Shared parts of the FP32 strip-walk kernels (euler_force_walk.cuh,
// euler_walk2d.cuh): one cooperative launch advances a field K steps, warps
// walk strips of the field row by row, a bounded grid barrier separates
// dependent phases.
//
// A walk holds a strip in the lanes of one warp, lane l the pair of cells
// (2l, 2l + 1) as f32x2 values, and moves along an axis one row at a time, so
// everything carried from row to row stays in registers and everything
// exchanged between columns is a warp shuffle: no tile, no CTA barrier.
#pragma once
#include <cstdint>

#include "euler_sweep.cuh"
#include "grid_sync.cuh"
#include "pair_math.cuh"
#include "tma.cuh"

namespace ripple {

constexpr int kWalkWarps = 16;  // warps per CTA, one CTA per SM
constexpr int kWalkUse = 60;   // columns updated by a walk that works along x too (of the 64 its lanes hold)

// Arguments of a multi-step walk launch.
struct WalkStep {
    float* buf[2];         // (FP64 tiles: doubles)
    FieldCtl* ctl;
    FieldGeom g;
    double cfl, gamma;
    double inv_dx[3];
    double dx_cfl[3];      // dx / cfl: dx / dt is that times the largest wave-speed sum
    float gamma_f, gm1_f, inv_dx_f[3];
    int bc;
    int K;                 // steps of this launch
    int cur;               // buffer holding the state at the start of the launch
    int slot;              // wave-speed ring slot of that state
    int first;             // the first step of a call: t = dt instead of t += dt
    int strips, rows, segs;     // in-plane walks: strips of columns, segments of `rows` rows
    int cols;                   // FP64 tiles: columns of a tile (rows: its rows)
    int zstrips, zrows, zsegs;  // walks along z (3D split step)
    unsigned spin_limit;   // polls of a barrier wait before it gives up
    unsigned* err;         // DEV_ERR_TIMEOUT when a barrier wait ran out
};

// The launch's grid barriers count up ctl->bar[0] (grid_sync.cuh); the last CTA
// to leave the kernel sets the barrier's and the units' words back to zero, so
// a launch needs no reset before it.  (Every acquiring poll drops the SM's L1
// lines, which a second CTA on the SM would still be working on: 230 against
// 169 us a step for 4096^2 FORCE with two CTAs of 8 warps per SM.  One CTA of
// 16 has no such neighbour.)
// Every CTA calls this once, after its last barrier; one whose wait ran out too:
// it arrives at no further barrier, so the others' waits run out as well and
// the last of them leaves the words at zero for whatever is queued behind this
// launch before the host has seen the error.
__device__ __forceinline__ void walk_leave(FieldCtl* ctl)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&ctl->bar[1], 1u) == gridDim.x - 1) {
            ctl->bar[0] = 0u;
            ctl->bar[1] = 0u;
            for (int i = 0; i < 4; ++i) ctl->work[i] = 0u;
        }
    }
}

// The units of a phase: each warp of the launch first walks the unit of its
// own number (warps of different CTAs first, so few units spread over the
// SMs), the rest are handed out one at a time from ctl->work[phase % 4] (the
// next one is asked for before the current one is walked, so its latency is
// hidden).  Handing them out keeps the warps of an SM busy to the end of a
// phase: a scheduler favours its oldest warps, and with one long unit per
// warp the last ones run alone (4096^2 FORCE: one unit of 118 rows per warp
// 169 us a step, handed out by 24 rows 115 us).  The counter is not touched
// when every unit has a warp of its own: 2,400 atomics on one word take 3 us.
struct WalkUnits {
    unsigned* next;
    int units, lane, warps, u, got;
    __device__ __forceinline__ WalkUnits(FieldCtl* ctl, unsigned phase, int n, int lane_, int warp)
        : next(&ctl->work[phase & 3u]), units(n), lane(lane_), warps((int)gridDim.x * kWalkWarps),
          u(warp * (int)gridDim.x + (int)blockIdx.x), got(0)
    {
        // the counter of the next phase was last used three phases ago
        if (blockIdx.x == 0 && threadIdx.x == 0) ctl->work[(phase + 1u) & 3u] = 0u;
    }
    __device__ __forceinline__ bool any() const { return u < units; }
    // ask for the unit after u
    __device__ __forceinline__ void ask()
    {
        if (units > warps && lane == 0) got = (int)atomicAdd(next, 1u);
        __syncwarp();
    }
    __device__ __forceinline__ void advance()
    {
        u = units > warps ? warps + __shfl_sync(0xffffffffu, got, 0) : units;
    }
};

// Row (or plane) index of a walk that starts one row before the field or ends
// one row after it: the interior row whose copy the ghost row would be.
__device__ __forceinline__ int walk_map(int r, int n, int bc)
{
    if (bc == 0) return r < 0 ? r + n : r >= n ? r - n : r;
    return min(max(r, 0), n - 1);
}

// The lane's pair in the rows r, r + 1, ... of a walk, mapped as above: a
// pointer that advances by one row inside the field.
struct WalkRows {
    const float* base;  // row 0
    const float* p;     // row r
    long long stride;
    int r, n, bc;
    __device__ __forceinline__ void init(const float* b, long long st, int r0, int n_, int bc_)
    {
        base = b;
        stride = st;
        r = r0;
        n = n_;
        bc = bc_;
        p = b + walk_map(r0, n_, bc_) * st;
    }
    __device__ __forceinline__ void next()
    {
        ++r;
        p += stride;
        if (r <= 0 || r >= n) p = base + walk_map(r, n, bc) * stride;  // warp-uniform, at the field's ends
    }
};

// What a walk gathers from its new states, per column of the lane's pair:
// the largest wave-speed sum and whether every state was admissible.
struct WalkNew {
    float s0 = 0.f, s1 = 0.f;
    bool ok0 = true, ok1 = true;
    template <int DIM>
    __device__ __forceinline__ void add(const f2 (&qn)[DIM + 2], f2 gamma, f2 gm1, const f2 (&ivx)[3])
    {
        bool o0, o1;
        const f2 sw = wave_sum2<DIM>(qn, gamma, gm1, ivx, o0, o1);
        s0 = fmaxf(s0, sw.x);
        s1 = fmaxf(s1, sw.y);
        ok0 &= o0;
        ok1 &= o1;
    }
};

// Report the first non-admissible new state of a column (rare, out of line):
// rows r0 .. r1 - 1 along `axis` of the column at element pointer p (row r0).
template <int DIM>
static __device__ __noinline__ void walk_bad_cell(FieldCtl* ctl, float gamma, float gm1, const float* p,
                                                  long long stride, long long cstr, int axis, int x, int line, int r0,
                                                  int r1)
{
    for (int r = r0; r < r1; ++r, p += stride) {
        float q[DIM + 2];
        for (int m = 0; m < DIM + 2; ++m) q[m] = p[m * cstr];
        const float ivx[3] = {1.f, 1.f, 1.f};
        bool ok;
        wave_sum<float, DIM>(q, gamma, gm1, ivx, ok);
        if (!ok) {
            record_bad(ctl, BAD_CELL, x, axis == 1 ? r : line, axis == 1 ? line : r);
            break;
        }
    }
    atomicOr(&ctl->err, DEV_ERR_NUMERIC);
}

// Store the updated pair of cells (x, x + 1) at element pointer p; v0, v1: the
// cell belongs to this walk and the field; full (warp-uniform): v0 == v1.
template <int DIM, int LAYOUT>
__device__ __forceinline__ void walk_store(float* p, long long cs, const f2 (&q)[DIM + 2], bool v0, bool v1, bool full)
{
    constexpr int NC = DIM + 2;
    if (v1) {
        if constexpr (LAYOUT == LAYOUT_SOA) {
#pragma unroll
            for (int m = 0; m < NC; ++m) *reinterpret_cast<float2*>(p + m * cs) = make_float2(q[m].x, q[m].y);
        } else if constexpr (NC == 4) {
            *reinterpret_cast<float4*>(p) = make_float4(q[0].x, q[1].x, q[2].x, q[3].x);
            *reinterpret_cast<float4*>(p + 4) = make_float4(q[0].y, q[1].y, q[2].y, q[3].y);
        } else {
            float2* d = reinterpret_cast<float2*>(p);  // 40 bytes of an even cell: 8-byte aligned
            d[0] = make_float2(q[0].x, q[1].x);
            d[1] = make_float2(q[2].x, q[3].x);
            d[2] = make_float2(q[4].x, q[0].y);
            d[3] = make_float2(q[1].y, q[2].y);
            d[4] = make_float2(q[3].y, q[4].y);
        }
    }
    if (!full) {
        if (v0 && !v1) {
#pragma unroll
            for (int m = 0; m < NC; ++m) p[m * (LAYOUT == LAYOUT_SOA ? cs : 1)] = q[m].x;
        }
    }
}

// Copy the lane's own pair of cells at element pointer p into its part of a
// ring slot (asynchronously: this thread waits for its own copy groups before
// it reads the slot, and no other thread reads it).
__device__ __forceinline__ void cp_async8(void* dst, const void* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
template <int DIM, int LAYOUT>
__device__ __forceinline__ void walk_stage(float* slot, int lane, const float* p, long long cs)
{
    constexpr int NC = DIM + 2;
    if constexpr (LAYOUT == LAYOUT_SOA) {
#pragma unroll
        for (int m = 0; m < NC; ++m) cp_async8(slot + 64 * m + 2 * lane, p + m * cs);
    } else if constexpr (NC == 4) {
        cp_async16(slot + 8 * lane, p);
        cp_async16(slot + 8 * lane + 4, p + 4);
    } else {
#pragma unroll
        for (int i = 0; i < NC; ++i) cp_async8(slot + 2 * NC * lane + 2 * i, p + 2 * i);
    }
}
template <int DIM, int LAYOUT>
__device__ __forceinline__ void walk_read(const float* slot, int lane, f2 (&q)[DIM + 2])
{
    constexpr int NC = DIM + 2;
    if constexpr (LAYOUT == LAYOUT_SOA) {
#pragma unroll
        for (int m = 0; m < NC; ++m) q[m] = *reinterpret_cast<const f2*>(slot + 64 * m + 2 * lane);
    } else if constexpr (NC == 4) {
        const float4 a = *reinterpret_cast<const float4*>(slot + 8 * lane);
        const float4 b = *reinterpret_cast<const float4*>(slot + 8 * lane + 4);
        q[0] = f2{a.x, b.x}; q[1] = f2{a.y, b.y}; q[2] = f2{a.z, b.z}; q[3] = f2{a.w, b.w};
    } else {
        float w[2 * NC];
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            const float2 v = *reinterpret_cast<const float2*>(slot + 2 * NC * lane + 2 * i);
            w[2 * i] = v.x;
            w[2 * i + 1] = v.y;
        }
#pragma unroll
        for (int m = 0; m < NC; ++m) q[m] = f2{w[m], w[NC + m]};
    }
}

// The images along x of an updated pair in a strip at the field's x ends; p:
// element pointer of the pair in the output.
template <int DIM, int LAYOUT>
__device__ __forceinline__ void walk_ghost_x(float* p, long long cs, const f2 (&q)[DIM + 2], int x, int nx, int h,
                                             int bc, bool v0, bool v1)
{
    constexpr int NC = DIM + 2;
    constexpr int CST = LAYOUT == LAYOUT_SOA ? 1 : NC;
    const long long ms = LAYOUT == LAYOUT_SOA ? cs : 1;
    auto put = [&](bool second, int to) {  // the pair's first or second cell, `to` cells from the first
#pragma unroll
        for (int m = 0; m < NC; ++m) p[(long long)to * CST + m * ms] = second ? q[m].y : q[m].x;
    };
    if (bc == 0) {
        if (v0 && x < h) put(false, nx);
        if (v0 && x >= nx - h) put(false, -nx);
        if (v1 && x + 1 < h) put(true, nx + 1);
        if (v1 && x + 1 >= nx - h) put(true, 1 - nx);
    } else {
        // the edge cell into the h layers beyond it
        const bool hi1 = v1 && x + 1 == nx - 1;
        for (int e = 1; e <= h; ++e) {
            if (v0 && x == 0) put(false, -e);
            if (hi1 || (v0 && x == nx - 1)) put(hi1, e + (hi1 ? 1 : 0));
        }
    }
    __syncwarp();
}

// The images of a row's pairs along another axis, on which the row is number
// c of n (the same for the whole warp); stride: elements from row to row.
template <int DIM, int LAYOUT>
__device__ __forceinline__ void walk_ghost_rows(float* p, long long cs, const f2 (&q)[DIM + 2], int c, int n, int h,
                                                int bc, long long stride, bool v0, bool v1, bool full)
{
    if (bc == 0) {
        if (c < h) walk_store<DIM, LAYOUT>(p + n * stride, cs, q, v0, v1, full);
        if (c >= n - h) walk_store<DIM, LAYOUT>(p - n * stride, cs, q, v0, v1, full);
    } else {
        if (c == 0)
            for (int e = 1; e <= h; ++e) walk_store<DIM, LAYOUT>(p - e * stride, cs, q, v0, v1, full);
        if (c == n - 1)
            for (int e = 1; e <= h; ++e) walk_store<DIM, LAYOUT>(p + e * stride, cs, q, v0, v1, full);
    }
}

// CTA maximum of the new states' wave-speed sums into the next ring slot.
__device__ __forceinline__ void walk_reduce(FieldCtl* ctl, int slot, float smax, float* red)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) smax = fmaxf(smax, __shfl_xor_sync(0xffffffffu, smax, o));
    if (lane == 0) red[warp] = smax;
    __syncthreads();
    if (threadIdx.x == 0) {
        float m = red[0];
        for (int w = 1; w < kWalkWarps; ++w) m = fmaxf(m, red[w]);
        atomic_max_pos_double(&ctl->smax[slot], (double)m);
    }
}

}  // namespace ripple
