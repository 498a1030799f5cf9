// Launchers of the auxiliary Euler kernels and the layout scatter/gather.
#include "euler_aux.cuh"
#include "runtime.h"

namespace ripple {

// Blocks of 256 threads for `items` work items: at most eight per SM (`cap`).
static int blocks_for(unsigned long long items, int cap)
{
    const unsigned long long b = (items + 255) / 256;
    return (int)(b < 1 ? 1 : b < (unsigned long long)cap ? b : (unsigned long long)cap);
}

template <typename T, int DIM>
static cudaError_t prep_t(void* buf, FieldCtl* ctl, const FieldGeom& g, int bc, double gamma, const double inv_dx[3],
                          int slot, int cap, cudaStream_t s)
{
    constexpr int V = 16 / (int)sizeof(T);
    T* b = static_cast<T*>(buf);
    if (g.cell_stride == 1)
        euler_prep_kernel<T, DIM, V><<<blocks_for(row_items<V>(g).items, cap), 256, 0, s>>>(
            b, ctl, g, bc, gamma, inv_dx[0], inv_dx[1], inv_dx[2], slot);
    else
        euler_prep_kernel<T, DIM, 1><<<blocks_for(row_items<1>(g).items, cap), 256, 0, s>>>(
            b, ctl, g, bc, gamma, inv_dx[0], inv_dx[1], inv_dx[2], slot);
    return cudaGetLastError();
}

cudaError_t launch_prep(int dtype, int dim, void* buf, FieldCtl* ctl, const FieldGeom& g, int bc, double gamma,
                        const double inv_dx[3], int slot, int cap, cudaStream_t s)
{
    if (dtype == RIPPLE_F32)
        return dim == 2 ? prep_t<float, 2>(buf, ctl, g, bc, gamma, inv_dx, slot, cap, s)
                        : prep_t<float, 3>(buf, ctl, g, bc, gamma, inv_dx, slot, cap, s);
    return dim == 2 ? prep_t<double, 2>(buf, ctl, g, bc, gamma, inv_dx, slot, cap, s)
                    : prep_t<double, 3>(buf, ctl, g, bc, gamma, inv_dx, slot, cap, s);
}

cudaError_t launch_pad_nan(int dtype, void* b0, void* b1, const FieldGeom& g, int cap, cudaStream_t s)
{
    const long long cells = g.px * g.py * g.pz - (long long)g.n[0] * g.n[1] * g.n[2];
    const int grid = blocks_for((unsigned long long)cells, cap);
    if (dtype == RIPPLE_F32)
        pad_fill_nan_kernel<float><<<grid, 256, 0, s>>>(static_cast<float*>(b0), static_cast<float*>(b1), g);
    else pad_fill_nan_kernel<double><<<grid, 256, 0, s>>>(static_cast<double*>(b0), static_cast<double*>(b1), g);
    return cudaGetLastError();
}

template <typename T, int NC>
static cudaError_t totals_t(const void* buf, const FieldGeom& g, double* partials, int nblocks, FieldCtl* ctl,
                            cudaStream_t s)
{
    constexpr int V = 16 / (int)sizeof(T);
    const T* b = static_cast<const T*>(buf);
    if (g.cell_stride == 1)
        totals_kernel<T, NC, V><<<blocks_for(row_items<V>(g).items, nblocks), 256, 0, s>>>(b, g, partials, ctl);
    else totals_kernel<T, NC, 1><<<blocks_for(row_items<1>(g).items, nblocks), 256, 0, s>>>(b, g, partials, ctl);
    return cudaGetLastError();
}

cudaError_t launch_totals(int dtype, int ncomp, const void* buf, const FieldGeom& g, double* partials, int nblocks,
                          FieldCtl* ctl, cudaStream_t s)
{
    const bool f32 = dtype == RIPPLE_F32;  // Euler fields: four or five components
    if (ncomp == 4)
        return f32 ? totals_t<float, 4>(buf, g, partials, nblocks, ctl, s)
                   : totals_t<double, 4>(buf, g, partials, nblocks, ctl, s);
    return f32 ? totals_t<float, 5>(buf, g, partials, nblocks, ctl, s)
               : totals_t<double, 5>(buf, g, partials, nblocks, ctl, s);
}

template <typename T, int NC>
static cudaError_t copy_t(void* buf, const FieldGeom& g, void* dense, long long dc, long long dm, int dir, int cap,
                          cudaStream_t s)
{
    constexpr int V = 16 / (int)sizeof(T);
    T* b = static_cast<T*>(buf);
    T* d = static_cast<T*>(dense);
    // 16-byte accesses need every dense row on a 16-byte boundary: the array,
    // the row length and so the component distance (a 4,096^2 call, copies in and
    // out and the first padding fill: 422 us beside the steps before, 246 now)
    const bool vec = g.cell_stride == 1 && dc == 1 && g.n[0] % V == 0 && reinterpret_cast<uintptr_t>(dense) % 16 == 0;
    if (vec)
        interior_copy_kernel<T, NC, V><<<blocks_for(row_items<V>(g).items, cap), 256, 0, s>>>(b, g, d, dc, dm, dir);
    else
        interior_copy_kernel<T, NC, 1><<<blocks_for(row_items<1>(g).items, cap), 256, 0, s>>>(b, g, d, dc, dm, dir);
    return cudaGetLastError();
}

template <typename T>
static cudaError_t copy_n(int nc, void* buf, const FieldGeom& g, void* dense, long long dc, long long dm, int dir,
                          int cap, cudaStream_t s)
{
    switch (nc) {
        case 1: return copy_t<T, 1>(buf, g, dense, dc, dm, dir, cap, s);
        case 2: return copy_t<T, 2>(buf, g, dense, dc, dm, dir, cap, s);
        case 3: return copy_t<T, 3>(buf, g, dense, dc, dm, dir, cap, s);
        case 4: return copy_t<T, 4>(buf, g, dense, dc, dm, dir, cap, s);
        default: return copy_t<T, 5>(buf, g, dense, dc, dm, dir, cap, s);
    }
}

cudaError_t launch_interior_copy(int dtype, void* buf, const FieldGeom& g, void* dense, int dense_layout, int dir,
                                 int cap, cudaStream_t s)
{
    FieldGeom f = g;
    int nc = g.ncomp;
    long long dc = dense_layout == LAYOUT_SOA ? 1 : nc;
    long long dm = dense_layout == LAYOUT_SOA ? (long long)g.n[0] * g.n[1] * g.n[2] : 1;
    if (dense_layout == LAYOUT_AOS && g.cell_stride == nc && nc > 1 && (long long)g.n[0] * nc <= INT32_MAX &&
        (unsigned long long)g.n[0] * nc * g.n[1] * g.n[2] <= (1ull << 32)) {
        // records on both sides: rows of ncomp times as many single numbers
        f.n[0] = g.n[0] * nc;
        f.px = g.px * nc;
        f.lead = (g.lead + g.h) * nc - g.h;
        f.cell_stride = 1;
        f.comp_stride = 0;
        f.ncomp = nc = 1;
        dc = 1;
        dm = 0;
    }
    return dtype == RIPPLE_F32 ? copy_n<float>(nc, buf, f, dense, dc, dm, dir, cap, s)
                               : copy_n<double>(nc, buf, f, dense, dc, dm, dir, cap, s);
}

cudaError_t launch_group(int dtype, int op, const GroupItem* items, int n, long long blocks, cudaStream_t s)
{
    if (n <= 0 || blocks <= 0) return cudaSuccess;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    const unsigned grid = (unsigned)blocks;
    if (dtype == RIPPLE_F32) {
        if (op == GROUP_ADMIT_FILL) group_admit_fill_kernel<float><<<grid, 256, 0, s>>>(items, n);
        else if (op == GROUP_ADMIT_PREP) group_admit_prep_kernel<float><<<grid, 256, 0, s>>>(items, n);
        else group_pack_kernel<float><<<grid, 256, 0, s>>>(items, n);
    } else {
        if (op == GROUP_ADMIT_FILL) group_admit_fill_kernel<double><<<grid, 256, 0, s>>>(items, n);
        else if (op == GROUP_ADMIT_PREP) group_admit_prep_kernel<double><<<grid, 256, 0, s>>>(items, n);
        else group_pack_kernel<double><<<grid, 256, 0, s>>>(items, n);
    }
    return cudaGetLastError();
}

}  // namespace ripple
