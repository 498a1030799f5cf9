// One visit of one Fast Iterative Method tile (Section 7.4 benchmark; block
// FIM of Jeong & Whitaker), shared by the persistent single-problem solver
// and the batched iteration kernel of the serving runtime.
//
// Which tiles iteration k visits, and which buffer each tile lives in, is the
// business of a bookkeeping policy (per-tile flags or lists of active tiles,
// below).  An active tile is read into registers (its interior from the buffer
// it lives in, the faces of its neighbours from theirs), relaxed by sweeps of
// T <- min(T, G(T)) until no cell moves by tol, and written to its other
// buffer; a tile that did not converge stays active and a boundary layer that
// moved by tol or more activates the neighbour across that face.
//
// A solve follows one chain: a front crosses a tile one cell per sweep, and
// iterations follow each other, so what counts is the latency of a sweep and
// of what surrounds it, not the number of updates.  Hence:
//   * four cells per thread stay in registers for the whole visit; neighbours
//     in the warp come by shuffles, those in the thread from registers, and
//     only the layers between two warps pass through shared memory;
//   * in FP32 two sweeps run between two exchanges of those layers, so a CTA
//     barrier (which also decides convergence) is paid once per exchange;
//   * everything a visit reads is requested at once: both buffers' values with
//     the words that say which one counts, so the visit starts after one trip
//     to L2 instead of three;
//   * the FP32 update has no branches.
// (Before: cells in shared memory, five loads and a barrier per sweep.)
#pragma once
#include <cstdint>
#include <type_traits>

#include "field.cuh"

namespace ripple {

constexpr int kMaxSources = 16;

template <typename T>
__device__ __forceinline__ T ldcg_t(const T* p);
template <>
__device__ __forceinline__ float ldcg_t<float>(const float* p) { return __ldcg(p); }
template <>
__device__ __forceinline__ double ldcg_t<double>(const double* p) { return __ldcg(p); }

__device__ __forceinline__ float inf_t(float) { return __int_as_float(0x7f800000); }
__device__ __forceinline__ double inf_t(double) { return __longlong_as_double(0x7ff0000000000000ll); }

// Square root of the local solver: FP32 uses the hardware approximation
// (relative error about 2^-22, far inside the FP32 bar against Fast Marching);
// FP64 keeps the correctly rounded square root.
__device__ __forceinline__ float fim_sqrt(float x)
{
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ double fim_sqrt(double x) { return sqrt(x); }

__device__ __forceinline__ float fim_min3(float a, float b, float c)
{
    float r;  // one instruction on sm_100 and later
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Minimum of two values that are not negative (travel times and infinity): as
// integers, off the FP64 pipe.
__device__ __forceinline__ float fim_min(float a, float b) { return fmin(a, b); }
__device__ __forceinline__ double fim_min(double a, double b)
{
    const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
    return __longlong_as_double(x < y ? x : y);
}
__device__ __forceinline__ double fim_max(double a, double b)
{
    const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
    return __longlong_as_double(x < y ? y : x);
}

// Godunov upwind local solver in FP64: a[d] = smaller neighbour value along
// axis d, f = s * h.  It branches: a warp whose cells are all one-sided skips
// the roots, and FP64 issues at 1/64 of the FP32 rate (48 x 40 x 62: 3.6 ms a
// solve with the branches, 4.1 without).
template <int DIM>
__device__ __forceinline__ double godunov(double a0, double a1, double a2, double f)
{
    double x = fim_min(a0, a1), y = fim_max(a0, a1);
    if (DIM == 2) {
        const double d = a0 - a1;
        if (!(fabs(d) < f)) return x + f;
        return 0.5 * (a0 + a1 + fim_sqrt(2.0 * f * f - d * d));
    }
    const double z = fim_max(y, a2), m = fim_min(y, a2);
    y = fim_max(x, m);
    x = fim_min(x, m);
    double t = x + f;
    if (!(t > y)) return t;
    const double d = x - y;
    t = 0.5 * (x + y + fim_sqrt(2.0 * f * f - d * d));
    if (!(t > z)) return t;
    // 3 f^2 less the squared pairwise differences: no terms of size T^2 cancel
    const double dxz = x - z, dyz = y - z;
    const double disc = fmax(3.0 * f * f - (d * d + dxz * dxz + dyz * dyz), 0.0);
    return (x + y + z + fim_sqrt(disc)) * (1.0 / 3.0);
}

// min(v, G) in FP32, G the Godunov value of a cell whose value is v; ff2 = 2 f^2.
// Without branches: the candidates with one, two and three neighbours are all
// formed, and each further one counts while the next neighbour lies below the
// value so far (it is then the smaller one).
//   one: the smallest neighbour x plus f, rounded once, at any scale of f.  The
//       others square f and hold where f^2 is a normal number.
//   two: x + u, u the larger root of u^2 + (u - p)^2 = f^2, p the distance from
//       x to the second neighbour y;
//   three: x + u, u the larger root of u^2 + (u - p)^2 + (u - q)^2 = f^2, q the
//       distance from x to the third neighbour z.
// Only differences enter the roots, so nothing of size T^2 cancels.  Comparing
// with min(v, ...) passes over neighbours that are not below v, which could
// only give a candidate above v: infinite ones (their candidates may be NaN),
// and the cell's own value, which the shuffles return at a warp's edges.  f =
// inf (a cell that keeps its value) gives v.
// (A form with p clamped at f, so that the root covers one-sided cells too, is
// as fast but rounds them through the root: f/2 where f^2 vanishes, below 1e-19,
// and no value where it overflows, above 1e19.)
template <int DIM>
__device__ __forceinline__ float godunov_min(float a0, float a1, float a2, float f, float ff2, float v)
{
    const float lo = fmin(a0, a1), hi = fmax(a0, a1);
    if (DIM == 2) {
        const float p = hi - lo, two = fmaf(0.5f, p + fim_sqrt(fmaf(-p, p, ff2)), lo);
        const float m = fmin(v, lo + f);
        return hi < m ? fmin(m, two) : m;
    }
    const float x = fmin(lo, a2), z = fmax(hi, a2), y = fmax(lo, fmin(hi, a2));
    const float p = y - x, q = z - x;
    const float two = fmaf(0.5f, p + fim_sqrt(fmaf(-p, p, ff2)), x);
    // 3 f^2 - 2 (p^2 - p q + q^2)
    const float g = fmaf(p, q - p, -q * q), disc = fmaf(1.5f, ff2, g + g);
    const float three = fmaf(1.f / 3.f, p + q + fim_sqrt(disc), x);
    float m = fmin(v, x + f);
    m = y < m ? fmin(m, two) : m;
    return z < m ? fmin(m, three) : m;
}

template <int DIM>
struct EikTile {
    static constexpr int TS = DIM == 2 ? 32 : 8;
    static constexpr int CELLS = DIM == 2 ? TS * TS : TS * TS * TS;
    static constexpr int CPT = 4;           // cells per thread: rows (2D) or z layers (3D)
    static constexpr int NT = CELLS / CPT;  // threads per tile: 8 warps (2D), 4 warps (3D)
};
// Sweeps between two exchanges (2048^2 FP32: 1 1674, 2 1509, 4 1540 us).  FP64
// takes plain Jacobi sweeps: what the exchange costs is little beside a sweep's
// FP64 work, and a second sweep on old layers is work that does not help.
template <typename T>
constexpr int kFimInner = sizeof(T) == 8 ? 1 : 2;
// A visit ends unconverged after this many sweeps: visits are cheapest when
// almost all of them converge (2048^2 FP32: 1509 us at 96, 1700 at 64, 2826 at
// 48).  FP64: 64 and 48, six tile sides in 3D.
template <typename T, int DIM>
constexpr int kFimMaxSweeps = sizeof(T) == 8 ? (DIM == 2 ? 64 : 48) : (DIM == 2 ? 96 : 64);

// Per-problem state of the FIM iteration.  Two bookkeeping schemes use it:
//   flags (the batched runtime): act[3][ntiles] active flags and cur[2][ntiles]
//     buffer indices, every tile touched by every iteration;
//   lists (the single-problem solver): list[3][ntiles] of the tiles active in
//     each iteration (count[] of them, handed out through take[]), a packed
//     word per tile state[t] = ((k + 1) << 1) | buffer, where k is the last
//     iteration that visited the tile, and mark[t] = 1 + the last iteration
//     the tile was queued for (so a tile enters a list once).
template <typename T>
struct FimProblem {
    T* buf[2];         // the two buffers of the T field
    const T* slow;     // slowness field
    FieldGeom gT, gS;
    int ntx, nty, ntz, ntiles;
    int nsrc;
    int src[kMaxSources][3];
    double h, tol;
    unsigned* act;       // flags: [3][ntiles]
    unsigned char* cur;  // flags: [2][ntiles]
    unsigned* count;     // [3]: tiles activated for each iteration
    int* list;           // lists: [3][ntiles]
    unsigned* state;     // lists: [ntiles]
    unsigned* mark;      // lists: [ntiles]
    unsigned* take;      // lists: [3] next list entry to hand out
};

// Bookkeeping with per-tile flags: every tile is visited (cheaply, if
// inactive) by every iteration, which clears its flag of iteration k + 2 and
// carries its buffer index to iteration k + 1.
template <typename T>
struct FimFlagBook {
    const FimProblem<T>& a;
    long long k;
    __device__ unsigned char buf_of(int t) const { return __ldcg(&a.cur[(size_t)(k % 2) * a.ntiles + t]); }
    __device__ bool active(int t) const
    {
        const unsigned is_active = __ldcg(&a.act[(size_t)(k % 3) * a.ntiles + t]);
        if (threadIdx.x == 0) {
            a.act[(size_t)((k + 2) % 3) * a.ntiles + t] = 0u;
            if (!is_active) a.cur[(size_t)((k + 1) % 2) * a.ntiles + t] = buf_of(t);
        }
        return is_active != 0u;
    }
    __device__ void begin(int t, unsigned char cb) const
    {
        if (threadIdx.x == 0) a.cur[(size_t)((k + 1) % 2) * a.ntiles + t] = (unsigned char)(1 - cb);
    }
    __device__ void activate(int nb) const
    {
        if (atomicExch(&a.act[(size_t)((k + 1) % 3) * a.ntiles + nb], 1u) == 0u) atomicAdd(&a.count[(k + 1) % 3], 1u);
    }
};

// Bookkeeping with lists of active tiles: only listed tiles are visited.  A
// visit of iteration k moves the tile to its other buffer; readers in the same
// iteration still see the old one ((state >> 1) == k + 1 means "moved in this
// iteration"), readers of later iterations the new one.
template <typename T>
struct FimListBook {
    const FimProblem<T>& a;
    long long k;
    __device__ unsigned char buf_of(int t) const
    {
        const unsigned w = __ldcg(&a.state[t]);
        const unsigned char b = (unsigned char)(w & 1u);
        return (w >> 1) == (unsigned)(k + 1) ? (unsigned char)(b ^ 1u) : b;
    }
    __device__ bool active(int) const { return true; }
    // (a thread that reads the word after this still sees the old buffer)
    __device__ void begin(int t, unsigned char cb) const
    {
        if (threadIdx.x == 0) a.state[t] = ((unsigned)(k + 1) << 1) | (unsigned)(1 - cb);
    }
    __device__ void activate(int nb) const
    {
        const unsigned want = (unsigned)(k + 2);
        if (atomicMax(&a.mark[nb], want) < want) {
            const unsigned pos = atomicAdd(&a.count[(k + 1) % 3], 1u);
            a.list[(size_t)((k + 1) % 3) * a.ntiles + pos] = nb;
        }
    }
};

// Layers that pass between the warps of a tile, double-buffered by exchange.
template <typename T, int DIM>
struct FimSmem;
template <typename T>
struct FimSmem<T, 2> {
    T top[2][8][32], bot[2][8][32];  // first and last row of each warp
    unsigned chg[2][8][4];           // lanes whose cell c changed, per warp (FP64)
    unsigned side_mask, done;
};
template <typename T>
struct FimSmem<T, 3> {
    T zl[2][4][32];    // each warp's layer at the tile's middle in z
    T yl[2][4][4][8];  // each warp's rows at the tile's middle in y, [z][x]
    unsigned chg[2][4][4];  // lanes whose cell c changed, per warp (FP64)
    unsigned side_mask, done;
};

// Visit tile t of problem `a` in iteration k (all threads of the CTA call it)
// with the bookkeeping `book` (FimFlagBook or FimListBook).  Adds one tile
// visit and the Godunov updates performed to the counters.
// 2D: warp w holds rows 4w .. 4w + 3, lane x column x.  3D: warp w holds rows
// y = 4 (w & 1) + lane / 8, columns x = lane % 8, layers z = 4 (w >> 1) + 0 .. 3.
template <typename T, int DIM, class Book>
__device__ __forceinline__ void fim_visit_tile(FimSmem<T, DIM>& sm, const FimProblem<T>& a, int t, long long k,
                                               long long& visits, long long& updates, const Book& book)
{
    using C = EikTile<DIM>;
    constexpr int TS = C::TS, CPT = C::CPT, W = TS;  // W: lanes of one row
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const T INF = inf_t(T(0));
    const T tol = (T)a.tol;
    const FieldGeom& gT = a.gT;
    const FieldGeom& gS = a.gS;

    if (!book.active(t)) return;
    ++visits;
    const int bx = t % a.ntx, by = (t / a.ntx) % a.nty, bz = DIM == 3 ? t / (a.ntx * a.nty) : 0;
    const int lx = DIM == 2 ? lane : lane & 7;
    const int ly = DIM == 2 ? CPT * w : 4 * (w & 1) + (lane >> 3);
    const int lz = DIM == 2 ? 0 : CPT * (w >> 1);
    const int gx = bx * TS + lx, gy = by * TS + ly, gz = bz * TS + lz;
    const long long cstep = DIM == 2 ? gT.px : gT.px * gT.py;  // from one of the thread's cells to the next
    const long long id0 = geom_cell(gT, gx, gy, gz);
    const long long is0 = geom_cell(gS, gx, gy, gz) * gS.cell_stride;
    const long long sstep = (DIM == 2 ? gS.px : gS.px * gS.py) * gS.cell_stride;
    const int nrun = DIM == 2 ? gT.n[1] - gy : gT.n[2] - gz;  // cells of the run inside the grid
    const bool col = gx < gT.n[0] && (DIM == 2 || gy < gT.n[1]);
    const T* b0 = a.buf[0];
    const T* b1 = a.buf[1];

    // ---- everything the visit reads, in one go ----
    // neighbours outside the warps: x ghosts of the edge columns (one per cell),
    // the row or layer before the first cell of the run and after the last (the
    // edge warps only), 3D: y ghosts of the edge rows (one per cell)
    const bool xlo = lx == 0, xhi = lx == TS - 1;
    const int tx_nb = xlo ? (bx > 0 ? t - 1 : -1) : xhi ? (bx + 1 < a.ntx ? t + 1 : -1) : -1;
    const int run_tiles = DIM == 2 ? a.ntx : a.ntx * a.nty;  // tile distance along the run
    const bool r_lo = DIM == 2 ? w == 0 : w < 2, r_hi = DIM == 2 ? w == 7 : w >= 2;
    const int tr_nb = r_lo ? ((DIM == 2 ? by : bz) > 0 ? t - run_tiles : -1)
                      : r_hi ? ((DIM == 2 ? by + 1 < a.nty : bz + 1 < a.ntz) ? t + run_tiles : -1)
                             : -1;
    const bool ylo = DIM == 3 && (w & 1) == 0 && lane < 8, yhi = DIM == 3 && (w & 1) == 1 && lane >= 24;
    const int ty_nb = ylo ? (by > 0 ? t - a.ntx : -1) : yhi ? (by + 1 < a.nty ? t + a.ntx : -1) : -1;
    T v[CPT], v1[CPT], f[CPT], xg[CPT], xg1[CPT], yg[CPT], yg1[CPT];
#pragma unroll
    for (int c = 0; c < CPT; ++c) {
        const bool in = col && c < nrun;
        const long long id = id0 + c * cstep;
        v[c] = v1[c] = xg[c] = xg1[c] = yg[c] = yg1[c] = f[c] = INF;
        if (in) {
            v[c] = ldcg_t(b0 + id);
            v1[c] = ldcg_t(b1 + id);
            f[c] = a.slow[is0 + c * sstep];
        }
        if (in && tx_nb >= 0) {
            xg[c] = ldcg_t(b0 + id + (xlo ? -1 : 1));
            xg1[c] = ldcg_t(b1 + id + (xlo ? -1 : 1));
        }
        if (DIM == 3 && in && ty_nb >= 0) {
            yg[c] = ldcg_t(b0 + id + (ylo ? -gT.px : gT.px));
            yg1[c] = ldcg_t(b1 + id + (ylo ? -gT.px : gT.px));
        }
    }
    T rg = INF, rg1 = INF;
    if (col && tr_nb >= 0) {
        const long long id = r_lo ? id0 - cstep : id0 + CPT * cstep;
        rg = ldcg_t(b0 + id);
        rg1 = ldcg_t(b1 + id);
    }
    const unsigned char cb = book.buf_of(t);
    const bool xb = tx_nb >= 0 && book.buf_of(tx_nb) != 0, rb = tr_nb >= 0 && book.buf_of(tr_nb) != 0;
    const bool yb = DIM == 3 && ty_nb >= 0 && book.buf_of(ty_nb) != 0;
    book.begin(t, cb);
    T init[CPT];
#pragma unroll
    for (int c = 0; c < CPT; ++c) {
        if (cb) v[c] = v1[c];
        if (xb) xg[c] = xg1[c];
        if (yb) yg[c] = yg1[c];
        init[c] = v[c];
        f[c] = f[c] * (T)a.h;  // outside the grid: infinite, so the cell keeps its (infinite) value
    }
    if (rb) rg = rg1;
    // sources keep their value; in the first iteration they count as changed, so
    // that a source on a tile's edge reaches the tile beside it even when no
    // other cell of its tile does
    for (int q = 0; q < a.nsrc; ++q) {
        if (a.src[q][0] != gx || (DIM == 3 && a.src[q][1] != gy)) continue;
        const int c = DIM == 2 ? a.src[q][1] - gy : a.src[q][2] - gz;
#pragma unroll
        for (int e = 0; e < CPT; ++e)
            if (c == e) {
                f[e] = INF;
                if (k == 0) init[e] = INF;
            }
    }

    // ---- sweeps ----
    bool converged = false, moved = true;
    int sweeps = 0, par = 0;
    T lo = rg, hi = rg;  // the neighbours of the run's first and last cell
    // FP64: the lanes whose cell c changed in the last sweep.  A cell none of
    // whose neighbours changed keeps its value, and a warp skips a row or layer
    // of such cells: FP64 arithmetic is what a sweep costs.
    constexpr bool F64 = std::is_same<T, double>::value;
    unsigned chg[CPT];
    unsigned done = 0;  // cells this warp has updated (FP64)
    T ff2[CPT];  // 2 f^2 (FP32)
#pragma unroll
    for (int c = 0; c < CPT; ++c) {
        chg[c] = 0xffffffffu;
        ff2[c] = T(2) * f[c] * f[c];
    }
    for (;;) {
        // exchange the layers between warps; the barrier also tells whether any
        // cell has moved since the last one
        if (DIM == 2) {
            if constexpr (DIM == 2) {
                sm.top[par][w][lane] = v[0];
                sm.bot[par][w][lane] = v[CPT - 1];
            }
        } else {
            if constexpr (DIM == 3) {
                sm.zl[par][w][lane] = r_lo ? v[CPT - 1] : v[0];
                if ((w & 1) == 0 ? lane >= 24 : lane < 8) {
#pragma unroll
                    for (int c = 0; c < CPT; ++c) sm.yl[par][w][c][lx] = v[c];
                }
            }
        }
        if (F64 && lane == 0) {
#pragma unroll
            for (int c = 0; c < CPT; ++c) sm.chg[par][w][c] = chg[c];
        }
        if (!__syncthreads_or(moved ? 1 : 0)) {
            converged = true;
            break;
        }
        if (sweeps >= kFimMaxSweeps<T, DIM>) break;
        if constexpr (DIM == 2) {
            if (w > 0) lo = sm.bot[par][w - 1][lane];
            if (w < 7) hi = sm.top[par][w + 1][lane];
        } else {
            if (r_lo) hi = sm.zl[par][w ^ 2][lane];
            else lo = sm.zl[par][w ^ 2][lane];
            if ((w & 1) == 0 ? lane >= 24 : lane < 8) {
#pragma unroll
                for (int c = 0; c < CPT; ++c) yg[c] = sm.yl[par][w ^ 1][c][lx];
            }
        }
        moved = false;
        if constexpr (F64) {
            // cells with a neighbour that changed (warp-uniform masks)
            unsigned need[CPT];
#pragma unroll
            for (int c = 0; c < CPT; ++c) {
                const unsigned m = chg[c];
                if (DIM == 2) {
                    need[c] = m << 1 | m >> 1;
                } else {
                    need[c] = (m << 1 & 0xfefefefeu) | (m >> 1 & 0x7f7f7f7fu) | m << 8 | m >> 8;
                    const unsigned o = sm.chg[par][w ^ 1][c];
                    need[c] |= (w & 1) == 0 ? o << 24 : o >> 24;
                }
                if (c > 0) need[c] |= chg[c == 0 ? 0 : c - 1];
                if (c < CPT - 1) need[c] |= chg[c == CPT - 1 ? c : c + 1];
            }
            if (DIM == 2) {
                if (w > 0) need[0] |= sm.chg[par][w - 1][CPT - 1];
                if (w < 7) need[CPT - 1] |= sm.chg[par][w + 1][0];
            } else if (r_lo) {
                need[CPT - 1] |= sm.chg[par][w ^ 2][0];
            } else {
                need[0] |= sm.chg[par][w ^ 2][CPT - 1];
            }
            T nv[CPT];
#pragma unroll
            for (int c = 0; c < CPT; ++c) {
                nv[c] = v[c];
                chg[c] = 0u;
                if (need[c] == 0u) continue;
                done += __popc(need[c]);
                T l = __shfl_up_sync(0xffffffffu, v[c], 1, W), r = __shfl_down_sync(0xffffffffu, v[c], 1, W);
                if (xlo) l = xg[c];
                if (xhi) r = xg[c];
                const T below = c == 0 ? lo : v[c == 0 ? 0 : c - 1], above = c == CPT - 1 ? hi : v[c == CPT - 1 ? c : c + 1];
                const T ax = fim_min(l, r), ar = fim_min(below, above);
                T ay = INF;
                if (DIM == 3) {
                    const T u = __shfl_up_sync(0xffffffffu, v[c], 8), d = __shfl_down_sync(0xffffffffu, v[c], 8);
                    ay = fim_min(lane < 8 ? yg[c] : u, lane >= 24 ? yg[c] : d);
                }
                bool down = false;
                if (need[c] >> lane & 1u) {
                    const T g = DIM == 2 ? godunov<2>(ax, ar, INF, f[c]) : godunov<3>(ax, ay, ar, f[c]);
                    down = g < v[c];
                    if (down) {
                        moved |= v[c] - g >= tol;
                        nv[c] = g;
                    }
                }
                chg[c] = __ballot_sync(0xffffffffu, down);
            }
#pragma unroll
            for (int c = 0; c < CPT; ++c) v[c] = nv[c];
        } else {
#pragma unroll
            for (int s = 0; s < kFimInner<T>; ++s) {
                T nv[CPT];
#pragma unroll
                for (int c = 0; c < CPT; ++c) {
                    // at the warp's edges the shuffle returns the cell's own value, which the
                    // solver passes over, and the ghost is the third operand (infinite elsewhere)
                    const T l = __shfl_up_sync(0xffffffffu, v[c], 1, W), r = __shfl_down_sync(0xffffffffu, v[c], 1, W);
                    const T below = c == 0 ? lo : v[c == 0 ? 0 : c - 1], above = c == CPT - 1 ? hi : v[c == CPT - 1 ? c : c + 1];
                    if constexpr (DIM == 2) {
                        nv[c] = godunov_min<2>(fim_min3(l, r, xg[c]), fmin(below, above), INF, f[c], ff2[c], v[c]);
                    } else {
                        const T u = __shfl_up_sync(0xffffffffu, v[c], 8), d = __shfl_down_sync(0xffffffffu, v[c], 8);
                        nv[c] = godunov_min<3>(fim_min3(l, r, xg[c]), fim_min3(u, d, yg[c]), fmin(below, above), f[c],
                                               ff2[c], v[c]);
                    }
                    moved |= v[c] - nv[c] >= tol;
                }
#pragma unroll
                for (int c = 0; c < CPT; ++c) v[c] = nv[c];
            }
        }
        sweeps += kFimInner<T>;
        par ^= 1;
    }
    // ---- write back; boundary-layer changes activate neighbours ----
    if (tid == 0) sm.side_mask = sm.done = 0u;
    __syncthreads();
    if (F64 && lane == 0) atomicAdd(&sm.done, done);
    T* out = a.buf[1 - cb];
    bool any = false, first = false, last = false;
#pragma unroll
    for (int c = 0; c < CPT; ++c) {
        if (col && c < nrun) out[id0 + c * cstep] = v[c];
        const bool ch = init[c] - v[c] >= tol;
        any |= ch;
        if (c == 0) first = ch && r_lo;
        if (c == CPT - 1) last = ch && r_hi;
    }
    const unsigned by_lane = __ballot_sync(0xffffffffu, any);
    const bool b_first = __any_sync(0xffffffffu, first), b_last = __any_sync(0xffffffffu, last);
    if (lane == 0) {
        unsigned m;  // bits: x low, x high, y low, y high, z low, z high
        if (DIM == 2) {
            m = (by_lane & 1u) | ((by_lane >> 31) << 1) | (b_first ? 4u : 0u) | (b_last ? 8u : 0u);
        } else {
            m = ((by_lane & 0x01010101u) ? 1u : 0u) | ((by_lane & 0x80808080u) ? 2u : 0u) |
                ((w & 1) == 0 && (by_lane & 0xffu) ? 4u : 0u) | ((w & 1) == 1 && (by_lane >> 24) ? 8u : 0u) |
                (b_first ? 16u : 0u) | (b_last ? 32u : 0u);
        }
        if (m) atomicOr(&sm.side_mask, m);
    }
    __syncthreads();
    if (tid <= 2 * DIM) {
        // one thread per tile that may become active: this one, then across each side
        const unsigned m = sm.side_mask;
        const int side = tid - 1, axis = side >> 1;
        int nb = -1;
        if (tid == 0) nb = converged ? -1 : t;
        else if (m >> side & 1u) {
            const int pos = axis == 0 ? bx : axis == 1 ? by : bz, cnt = axis == 0 ? a.ntx : axis == 1 ? a.nty : a.ntz;
            const int dist = axis == 0 ? 1 : axis == 1 ? a.ntx : a.ntx * a.nty;
            if (side & 1) nb = pos + 1 < cnt ? t + dist : -1;
            else nb = pos > 0 ? t - dist : -1;
        }
        if (nb >= 0) book.activate(nb);
    }
    updates += F64 ? (long long)sm.done : (long long)sweeps * C::CELLS;
    __syncthreads();
}

}  // namespace ripple
