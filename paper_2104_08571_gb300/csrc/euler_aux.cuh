// Auxiliary kernels of the Euler path: the first padding fill + wave-speed
// reduction of a freshly uploaded state, the FP64 compensated conserved
// totals, and the interior scatter/gather used by upload and download.
#pragma once
#include <cstdint>

#include "euler_sweep.cuh"
#include "field.cuh"

namespace ripple {

// Read the conserved state of interior cell (i, j, k).
template <typename T, int DIM>
__device__ __forceinline__ void load_cell(const T* __restrict__ buf, const FieldGeom& g, int i, int j, int k,
                                          T (&q)[DIM + 2])
{
    const long long base = geom_cell(g, i, j, k) * g.cell_stride;
#pragma unroll
    for (int m = 0; m < DIM + 2; ++m) q[m] = buf[base + (long long)m * g.comp_stride];
}

__device__ __forceinline__ void cell_coords(const FieldGeom& g, long long lin, int& i, int& j, int& k)
{
    i = (int)(lin % g.n[0]);
    const long long r = lin / g.n[0];
    j = (int)(r % g.n[1]);
    k = (int)(r / g.n[1]);
}

// The interior of a field as items of V x-adjacent cells, numbered along rows:
// item it covers cells x .. x + V - 1 of row (y, z); at most 2^32 items, so
// the divisions are 32-bit (the 64-bit ones of a cell-per-item loop took more
// instructions than everything else in these kernels).
struct RowItems {
    unsigned per_row;
    unsigned long long items;
};
template <int V>
__host__ __device__ inline RowItems row_items(const FieldGeom& g)
{
    const unsigned p = (unsigned)((g.n[0] + V - 1) / V);
    return RowItems{p, (unsigned long long)p * (unsigned)g.n[1] * (unsigned)g.n[2]};
}
template <int V>
__device__ __forceinline__ void row_item(const FieldGeom& g, const RowItems& r, unsigned it, int& x, int& y, int& z,
                                         unsigned& row)
{
    row = it / r.per_row;
    x = (int)(it - row * r.per_row) * V;
    z = g.ndim == 3 ? (int)(row / (unsigned)g.n[1]) : 0;
    y = g.ndim == 3 ? (int)(row - (unsigned)z * (unsigned)g.n[1]) : (int)row;
}
// V consecutive elements by 16-byte accesses (V = 1: one element)
template <typename T, int V>
struct alignas(sizeof(T) * V) Vec {
    T v[V];
};

// set_boundary + set_wavespeeds + MaxReducer on the current buffer (used once
// after an upload or a change of boundary condition / gamma / dx; the sweep
// itself keeps both up to date afterwards).  The last block to finish moves
// the maximum into ring slot `slot` and clears the other two, so the launch
// needs no reset before it.  V cells of an SoA row per item (rows start on 16
// bytes and are padded to them, so the last item may read padding).
template <typename T, int DIM, int V>
__global__ void __launch_bounds__(256) euler_prep_kernel(T* __restrict__ buf, FieldCtl* __restrict__ ctl,
                                                         const FieldGeom g, int bc, double gamma, double idx0,
                                                         double idx1, double idx2, int slot)
{
    constexpr int NC = DIM + 2;
    const T gm = (T)gamma, gm1 = (T)(gamma - 1.0);
    const T inv_dx[3] = {(T)idx0, (T)idx1, (T)idx2};
    const RowItems ri = row_items<V>(g);
    T smax = T(0);
    bool bad = false;
    for (unsigned long long it = blockIdx.x * 256ull + threadIdx.x; it < ri.items; it += gridDim.x * 256ull) {
        int x, y, z;
        unsigned row;
        row_item<V>(g, ri, (unsigned)it, x, y, z, row);
        const long long base = geom_cell(g, x, y, z) * g.cell_stride;
        Vec<T, V> q[NC];
#pragma unroll
        for (int m = 0; m < NC; ++m)
            q[m] = *reinterpret_cast<const Vec<T, V>*>(buf + base + (long long)m * g.comp_stride);
        const bool near = y < g.h || y >= g.n[1] - g.h || (DIM == 3 && (z < g.h || z >= g.n[2] - g.h)) || x < g.h ||
                          x + V > g.n[0] - g.h;
#pragma unroll
        for (int c = 0; c < V; ++c) {
            if (V > 1 && x + c >= g.n[0]) break;
            T qc[NC];
#pragma unroll
            for (int m = 0; m < NC; ++m) qc[m] = q[m].v[c];
            bool ok;
            smax = fmax(smax, wave_sum<T, DIM>(qc, gm, gm1, inv_dx, ok));
            if (!ok) { bad = true; record_bad(ctl, BAD_INPUT, x + c, y, z); }
            if (near) write_ghost_images<T, DIM>(buf, g, bc, x + c, y, z, qc);
        }
    }
    __shared__ double red[8];
    double v = (double)smax;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int any_bad = __syncthreads_or(bad ? 1 : 0);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double m = 0.0;
        for (int w = 0; w < 8; ++w) m = fmax(m, red[w]);
        atomic_max_pos_double(&ctl->pmax, m);
        if (any_bad) atomicOr(&ctl->err, DEV_ERR_NUMERIC);
        __threadfence();
        if (atomicAdd(&ctl->done, 1u) == gridDim.x - 1) {
            __threadfence();
            ctl->smax[slot] = atomicExch(&ctl->pmax, 0ull);
            ctl->smax[(slot + 1) % 3] = 0ull;
            ctl->smax[(slot + 2) % 3] = 0ull;
            ctl->done = 0u;
        }
    }
}

// Quiet NaN in every padded cell outside the interior (all components) of both
// buffers.  The sweep rewrites the face ghosts each step; edge and corner
// ghosts and the alignment padding stay NaN, so a stencil item that reaches
// beyond the ghost layers carries NaN, which the admissibility minimum
// ignores.  Items: the cells left and right of the interior of every row,
// then the rest of the rows above and below it.
template <typename T>
__global__ void __launch_bounds__(256) pad_fill_nan_kernel(T* __restrict__ b0, T* __restrict__ b1, const FieldGeom g)
{
    const T qnan = (T)__int_as_float(0x7fc00000);
    const long long rows = g.py * g.pz, side = g.px - g.n[0];
    const int lo = g.lead + g.h;
    auto fill = [&](long long x, long long row) {
        const long long e = (row * g.px + x) * g.cell_stride;
        for (int m = 0; m < g.ncomp; ++m) b0[e + (long long)m * g.comp_stride] = b1[e + (long long)m * g.comp_stride] = qnan;
    };
    const long long t0 = blockIdx.x * 256ll + threadIdx.x, stride = gridDim.x * 256ll;
    for (long long i = t0; i < rows * side; i += stride) {
        const long long row = i / side, c = i % side;
        fill(c < lo ? c : c + g.n[0], row);
    }
    const long long h2 = 2 * g.h, in_rows = g.ndim == 3 ? g.n[2] * h2 : h2;  // y ghost rows of the inner planes
    const long long out_rows = g.ndim == 3 ? h2 * g.py : 0;                   // rows of the z ghost planes
    for (long long i = t0; i < (in_rows + out_rows) * g.n[0]; i += stride) {
        const long long r = i / g.n[0], x = lo + i % g.n[0];
        long long row;
        if (r < in_rows) {
            const long long pl = r / h2, k = r % h2, py = k < g.h ? k : k + g.n[1];
            row = (g.ndim == 3 ? (pl + g.h) * g.py : 0) + py;
        } else {
            const long long k = (r - in_rows) / g.py, py = (r - in_rows) % g.py;
            row = (k < g.h ? k : k + g.n[2]) * g.py + py;
        }
        fill(x, row);
    }
}

// Neumaier (improved Kahan-Babuska) compensated accumulation in FP64.
struct Neumaier {
    double s, c;
    __device__ void add(double x)
    {
        const double t = s + x;
        if (fabs(s) >= fabs(x)) c += (s - t) + x;
        else c += (x - t) + s;
        s = t;
    }
    __device__ void merge(const Neumaier& o)
    {
        add(o.s);
        c += o.c;
    }
};

// FP64 compensated sums of each component over the interior: a sum per thread,
// combined in a fixed order per block, partials[(block * NCOMP + m) * 2 + {0:
// sum, 1: compensation}]; the last block to finish combines the blocks' sums
// (one thread for 256 blocks, then the same fixed order), so the result does
// not depend on which block that is.  (A second launch with one thread per
// component walked the 304 partials one after the other: a 64^2 call of four
// steps with statistics 190 us, now 98.)
template <int NCOMP>
__device__ __forceinline__ void totals_block(Neumaier (&acc)[NCOMP], double (*sh)[NCOMP][2], Neumaier& out)
{
#pragma unroll
    for (int m = 0; m < NCOMP; ++m) {
        for (int o = 16; o > 0; o >>= 1) {
            Neumaier other{__shfl_down_sync(0xffffffffu, acc[m].s, o), __shfl_down_sync(0xffffffffu, acc[m].c, o)};
            acc[m].merge(other);
        }
    }
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0)
        for (int m = 0; m < NCOMP; ++m) {
            sh[w][m][0] = acc[m].s;
            sh[w][m][1] = acc[m].c;
        }
    __syncthreads();
    out = Neumaier{0.0, 0.0};
    if (threadIdx.x < NCOMP)
        for (int ww = 0; ww < 8; ++ww) out.merge(Neumaier{sh[ww][threadIdx.x][0], sh[ww][threadIdx.x][1]});
}

template <typename T, int NCOMP, int V>
__global__ void __launch_bounds__(256) totals_kernel(const T* __restrict__ buf, const FieldGeom g,
                                                     double* __restrict__ partials, FieldCtl* __restrict__ ctl)
{
    Neumaier acc[NCOMP];
#pragma unroll
    for (int m = 0; m < NCOMP; ++m) acc[m] = Neumaier{0.0, 0.0};
    const RowItems ri = row_items<V>(g);
    for (unsigned long long it = blockIdx.x * 256ull + threadIdx.x; it < ri.items; it += gridDim.x * 256ull) {
        int x, y, z;
        unsigned row;
        row_item<V>(g, ri, (unsigned)it, x, y, z, row);
        const long long base = geom_cell(g, x, y, z) * g.cell_stride;
        Vec<T, V> q[NCOMP];
#pragma unroll
        for (int m = 0; m < NCOMP; ++m)
            q[m] = *reinterpret_cast<const Vec<T, V>*>(buf + base + (long long)m * g.comp_stride);
#pragma unroll
        for (int c = 0; c < V; ++c) {
            if (V > 1 && x + c >= g.n[0]) break;
#pragma unroll
            for (int m = 0; m < NCOMP; ++m) acc[m].add((double)q[m].v[c]);
        }
    }
    __shared__ double sh[8][NCOMP][2];
    __shared__ bool last;
    Neumaier b;
    totals_block<NCOMP>(acc, sh, b);
    if (threadIdx.x < NCOMP) {
        double* p = partials + ((long long)blockIdx.x * NCOMP + threadIdx.x) * 2;
        p[0] = b.s;
        p[1] = b.c;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&ctl->done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
#pragma unroll
    for (int m = 0; m < NCOMP; ++m) {
        acc[m] = Neumaier{0.0, 0.0};
        for (unsigned k = threadIdx.x; k < gridDim.x; k += 256u) {
            const double* p = partials + ((long long)k * NCOMP + m) * 2;
            acc[m].merge(Neumaier{__ldcg(p), __ldcg(p + 1)});
        }
    }
    totals_block<NCOMP>(acc, sh, b);
    if (threadIdx.x < NCOMP) ctl->totals[threadIdx.x] = b.s + b.c;
    if (threadIdx.x == 0) ctl->done = 0u;
}

// Interior copy between a dense array and the padded field, both given by the
// distance from cell to cell and from component to component (g: the field's,
// dc and dm: the dense array's).  dir = 0: dense -> field (upload), dir = 1:
// field -> dense (download).  V > 1: both component-major and every dense row
// on a 16-byte boundary.
template <typename T, int NC, int V>
__global__ void __launch_bounds__(256) interior_copy_kernel(T* __restrict__ buf, const FieldGeom g,
                                                            T* __restrict__ dense, long long dc, long long dm, int dir)
{
    const RowItems ri = row_items<V>(g);
    for (unsigned long long it = blockIdx.x * 256ull + threadIdx.x; it < ri.items; it += gridDim.x * 256ull) {
        int x, y, z;
        unsigned row;
        row_item<V>(g, ri, (unsigned)it, x, y, z, row);
        T* f = buf + geom_cell(g, x, y, z) * g.cell_stride;
        T* d = dense + ((long long)row * g.n[0] + x) * dc;
        Vec<T, V> q[NC];
        if (dir == 0) {
#pragma unroll
            for (int m = 0; m < NC; ++m) q[m] = *reinterpret_cast<const Vec<T, V>*>(d + m * dm);
#pragma unroll
            for (int m = 0; m < NC; ++m) *reinterpret_cast<Vec<T, V>*>(f + m * g.comp_stride) = q[m];
        } else {
#pragma unroll
            for (int m = 0; m < NC; ++m) q[m] = *reinterpret_cast<const Vec<T, V>*>(f + m * g.comp_stride);
#pragma unroll
            for (int m = 0; m < NC; ++m) *reinterpret_cast<Vec<T, V>*>(d + m * dm) = q[m];
        }
    }
}


// ---------------------------------------------------------------------------
// Grouped admission and download of the batch runtime: one launch covers every
// instance of a group, each instance owning a contiguous run of blocks
// (GroupItem::blk[pass] = its first block in launch `pass`; instances with no
// blocks in a launch repeat the next instance's value).
// ---------------------------------------------------------------------------
__device__ __forceinline__ int group_find(const GroupItem* __restrict__ items, int n, int pass, long long b)
{
    // last item whose first block is <= b
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (items[mid].blk[pass] <= b) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ bool padded_inside(const FieldGeom& g, long long c, int& i, int& j, int& k)
{
    const long long x = c % g.px, r = c / g.px;
    const long long y = r % g.py, z = r / g.py;
    i = (int)(x - g.lead - g.h);
    j = (int)(y - g.h);
    k = g.ndim < 3 ? 0 : (int)(z - g.h);
    return i >= 0 && i < g.n[0] && j >= 0 && j < g.n[1] && (g.ndim < 3 || (k >= 0 && k < g.n[2]));
}

// Admission, launch 0 (padded cells of buffer 0): interior cells from the dense
// component-major input held in buffer 1, every other cell quiet NaN; the
// first block of an instance also clears its slot (control block, status,
// counters).  Eikonal instances own one block, which only clears the slot.
template <typename T>
__global__ void __launch_bounds__(256) group_admit_fill_kernel(const GroupItem* __restrict__ items, int n)
{
    const int it = group_find(items, n, 0, blockIdx.x);
    const GroupItem& d = items[it];
    const long long local = blockIdx.x - d.blk[0];
    if (local == 0) {
        unsigned* w = reinterpret_cast<unsigned*>(d.ctl);
        for (int q = threadIdx.x; q < (int)(sizeof(FieldCtl) / sizeof(unsigned)); q += blockDim.x) w[q] = 0u;
        if (threadIdx.x == 0) *d.status = 0ull;
        if (threadIdx.x < 3) d.counters[threadIdx.x] = 0;
    }
    if (!d.euler) return;
    const FieldGeom& g = d.g;
    T* buf = static_cast<T*>(d.buf);
    const T* dense = static_cast<const T*>(d.other);
    const long long cells = g.px * g.py * g.pz;
    const long long total = (long long)g.n[0] * g.n[1] * g.n[2];
    const T qnan = (T)__int_as_float(0x7fc00000);
    const long long c0 = local * kGroupCellsPerBlock;
    for (long long c = c0 + threadIdx.x; c < c0 + kGroupCellsPerBlock && c < cells; c += blockDim.x) {
        int i, j, k;
        const bool inside = padded_inside(g, c, i, j, k);
        const long long lin = ((long long)k * g.n[1] + j) * g.n[0] + i;
        for (int m = 0; m < g.ncomp; ++m)
            buf[c * g.cell_stride + (long long)m * g.comp_stride] = inside ? dense[(long long)m * total + lin] : qnan;
    }
}

// Admission, launch 1 (padded cells again): on buffer 0 the boundary images
// of each interior cell, the largest wave-speed sum (ring slot 0) and the
// admissibility check of the input; on buffer 1 quiet NaN outside the
// interior.  Runs after launch 0 (buffer 1's dense input has been read).
template <typename T>
__global__ void __launch_bounds__(256) group_admit_prep_kernel(const GroupItem* __restrict__ items, int n)
{
    const int it = group_find(items, n, 1, blockIdx.x);
    const GroupItem& d = items[it];
    const long long local = blockIdx.x - d.blk[1];
    const FieldGeom& g = d.g;
    T* buf = static_cast<T*>(d.buf);
    T* other = static_cast<T*>(d.other);
    const T gm = (T)d.gamma, gm1 = (T)(d.gamma - 1.0);
    const T inv_dx[3] = {(T)d.inv_dx0, (T)d.inv_dx1, (T)0};
    const long long cells = g.px * g.py * g.pz;
    const T qnan = (T)__int_as_float(0x7fc00000);
    T smax = T(0);
    bool bad = false;
    const long long c0 = local * kGroupCellsPerBlock;
    for (long long c = c0 + threadIdx.x; c < c0 + kGroupCellsPerBlock && c < cells; c += blockDim.x) {
        int i, j, k;
        if (!padded_inside(g, c, i, j, k)) {
            for (int m = 0; m < g.ncomp; ++m) other[c * g.cell_stride + (long long)m * g.comp_stride] = qnan;
            continue;
        }
        T q[4];
        load_cell<T, 2>(buf, g, i, j, k, q);
        bool ok;
        smax = fmax(smax, wave_sum<T, 2>(q, gm, gm1, inv_dx, ok));
        if (!ok) { bad = true; record_bad(d.ctl, BAD_INPUT, i, j, k); }
        write_ghost_images<T, 2>(buf, g, d.bc, i, j, k, q);
    }
    __shared__ double red[8];
    double v = (double)smax;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int any_bad = __syncthreads_or(bad ? 1 : 0);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double m = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = fmax(m, red[w]);
        atomic_max_pos_double(&d.ctl->smax[0], m);
        if (any_bad) atomicOr(&d.ctl->err, DEV_ERR_NUMERIC);
    }
}

// Download: the interior of each instance's result buffer into its dense
// component-major stage (interior cells, blk[0]).
template <typename T>
__global__ void __launch_bounds__(256) group_pack_kernel(const GroupItem* __restrict__ items, int n)
{
    const int it = group_find(items, n, 0, blockIdx.x);
    const GroupItem& d = items[it];
    const long long local = blockIdx.x - d.blk[0];
    const FieldGeom& g = d.g;
    const T* buf = static_cast<const T*>(d.buf);
    T* dense = static_cast<T*>(d.other);
    const long long total = (long long)g.n[0] * g.n[1] * g.n[2];
    const long long l0 = local * kGroupCellsPerBlock;
    for (long long lin = l0 + threadIdx.x; lin < l0 + kGroupCellsPerBlock && lin < total; lin += blockDim.x) {
        int i, j, k;
        cell_coords(g, lin, i, j, k);
        const long long base = geom_cell(g, i, j, k) * g.cell_stride;
        for (int m = 0; m < g.ncomp; ++m) dense[(long long)m * total + lin] = buf[base + (long long)m * g.comp_stride];
    }
}

}  // namespace ripple
