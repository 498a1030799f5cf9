// Fast Iterative Method eikonal solver (the paper's Section 7.4 benchmark,
// Jeong & Whitaker's block FIM) for |grad T| s = 1 on a Cartesian grid.
//
// Design (GB300-native, single persistent cooperative launch):
//   * the grid is cut into tiles (32 x 32 in 2D, 8 x 8 x 8 in 3D); an active
//     tile is relaxed in registers with its ghost faces (cross stencil, no
//     corners) by sweeps of the Godunov upwind update T <- min(T, G(T)) until
//     no cell moves by tol or more (fim_tile.cuh);
//   * tiles are double-buffered across the two buffers of the T field: an
//     active tile reads its interior and its neighbours' faces from the
//     buffer each tile currently lives in and writes the other one, so reads
//     and writes of an iteration never overlap and the result does not depend
//     on scheduling (deterministic);
//   * active-list update: a tile that did not converge stays active; a tile
//     whose boundary layer moved by tol or more activates the neighbour
//     across that face;
//   * iterations are separated by a bounded grid barrier (co-residency from
//     the cooperative launch); the run ends when no tile is active, or with
//     DEV_ERR_TIMEOUT when the iteration cap is reached (DEV_ERR_BARRIER when
//     a barrier wait runs out instead).
// Outside-domain neighbours are +inf; sources stay at 0.
//
// What bounds it: the chain of sweeps.  An iteration lasts as long as its
// longest visit (60 to 96 sweeps of about 0.15 us) plus 3 us of list, loads and
// barrier.  Measured (tol 1e-6, two sources, whole solve, before -> now): 2048^2
// 2250 -> 1410 us, 192^3 1900 -> 1320 us.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "fim_tile.cuh"
#include "grid_sync.cuh"
#include "resident.h"
#include "runtime.h"

namespace ripple {

constexpr int kFimCtasPerSm2D = 2;

// Arguments of the persistent single-problem solve beyond the problem itself.
struct EikArgs {
    long long max_iters;
    unsigned* bar;  // grid barrier: arrivals (zero at launch)
    unsigned spin_limit;  // polls of a barrier wait before it gives up
    FieldCtl* ctl;
};

struct EikScratch {
    size_t bytes = 0;
    void* mem = nullptr;
    int ntiles = 0;
};

// CTAs per SM the solve is compiled for.  2D: two, so that a thread may hold a
// visit's whole state (the compiler's own choice, 64 registers, ran 2048^2 in
// 1700 us, this 1415); 3D: six in FP32 (192^3: five 1345, six 1322, eight 1575 us).
template <typename T, int DIM>
constexpr int fim_min_ctas() { return DIM == 2 ? 2 : sizeof(T) == 4 ? 6 : 3; }

template <typename T, int DIM>
__global__ void __launch_bounds__(EikTile<DIM>::NT, fim_min_ctas<T, DIM>()) fim_kernel(const FimProblem<T> a, const EikArgs e)
{
    __shared__ FimSmem<T, DIM> sm;
    __shared__ int sflag[2];
    __shared__ unsigned s_next[2];
    const int tid = threadIdx.x;
    if (tid == 0) sflag[0] = 0;
    __syncthreads();

    long long visits = 0, updates = 0;
    long long k = 0;
    unsigned turn = 0;
    bool timed_out = false, barrier_out = false;
    for (;;) {
        // slots of iteration k - 1 are free: reset them for iteration k + 2
        if (blockIdx.x == 0 && tid == 0) {
            a.count[(k + 2) % 3] = 0u;
            a.take[(k + 2) % 3] = 0u;
        }
        // the active tiles of this iteration: each CTA takes the one of its own
        // number, the rest are handed out one at a time (asked for before the
        // visit in hand, so the answer is there after it)
        const int* list = a.list + (size_t)(k % 3) * a.ntiles;
        int t = __ldcg(list + blockIdx.x);  // read beside the count: the grid is no larger than the tiles
        const unsigned n = __ldcg(&a.count[k % 3]);
        const FimListBook<T> book{a, k};
        for (unsigned i = blockIdx.x; i < n;) {
            if (n > gridDim.x && tid == 0) s_next[turn & 1u] = gridDim.x + atomicAdd(&a.take[k % 3], 1u);
            fim_visit_tile<T, DIM>(sm, a, t, k, visits, updates, book);
            i = n > gridDim.x ? s_next[turn & 1u] : n;
            ++turn;
            if (i < n) t = __ldcg(list + i);
        }

        if (!grid_barrier(e.bar, (unsigned)(k + 1), e.spin_limit, sflag)) {
            barrier_out = true;
            break;
        }
        ++k;
        const unsigned remaining = __ldcg(&a.count[k % 3]);
        if (remaining == 0u) break;
        if (k >= e.max_iters) {
            timed_out = true;
            break;
        }
        // No second barrier: count[k % 3] and take[k % 3] are next reset in
        // iteration k + 1, which no CTA starts before every CTA has passed the
        // barrier that ends iteration k.
    }

    if (!timed_out && !barrier_out) {
        // consolidate: every tile's current values into buffer 0
        using C = EikTile<DIM>;
        constexpr int TS = C::TS;
        const FimListBook<T> book{a, k};
        for (int t = blockIdx.x; t < a.ntiles; t += gridDim.x) {
            if (book.buf_of(t) == 0) continue;
            const int bx = t % a.ntx, by = (t / a.ntx) % a.nty, bz = DIM == 3 ? t / (a.ntx * a.nty) : 0;
            for (int c = 0; c < C::CPT; ++c) {
                const int lin = tid + c * C::NT;
                const int x = lin % TS, y = (lin / TS) % TS, z = DIM == 3 ? lin / (TS * TS) : 0;
                const int gx = bx * TS + x, gy = by * TS + y, gz = bz * TS + z;
                if (gx < a.gT.n[0] && gy < a.gT.n[1] && gz < a.gT.n[2]) {
                    const long long id = geom_cell(a.gT, gx, gy, gz);
                    a.buf[0][id] = ldcg_t(&a.buf[1][id]);
                }
            }
        }
    }
    if (tid == 0) {
        atomicAdd((unsigned long long*)&e.ctl->counters[1], (unsigned long long)visits);
        atomicAdd((unsigned long long*)&e.ctl->counters[2], (unsigned long long)updates);
        if (blockIdx.x == 0) e.ctl->counters[0] = k;
        if (timed_out) atomicOr(&e.ctl->err, DEV_ERR_TIMEOUT);
        if (barrier_out) atomicOr(&e.ctl->err, DEV_ERR_BARRIER);
    }
}

// Initialise both buffers (+inf interior, 0 at sources) and the tiles of
// iteration 0 (those holding a source): the first list with every list's
// words (counts, marks, states, barrier) and the solver counters, or per-tile
// flags in zeroed memory (the batched runtime).
template <typename T>
__global__ void fim_init_kernel(const FimProblem<T> a, int ts, FieldCtl* ctl, unsigned* bar)
{
    const FieldGeom& g = a.gT;
    const T INF = inf_t(T(0));
    const unsigned nx = (unsigned)g.n[0], ny = (unsigned)g.n[1];
    const long long rows = (long long)ny * g.n[2];
    const unsigned long long total = (unsigned long long)nx * (unsigned long long)rows;
    for (unsigned long long lin = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; lin < total;
         lin += (unsigned long long)gridDim.x * blockDim.x) {
        const unsigned r = (unsigned)(lin / nx);
        const int i = (int)(lin - (unsigned long long)r * nx), j = (int)(r % ny), kk = (int)(r / ny);
        T v = INF;
        for (int q = 0; q < a.nsrc; ++q)
            if (a.src[q][0] == i && a.src[q][1] == j && (g.ndim == 2 || a.src[q][2] == kk)) v = T(0);
        const long long id = geom_cell(g, i, j, kk);
        a.buf[0][id] = v;
        a.buf[1][id] = v;
    }
    auto tile_of = [&](int q) {
        const int bx = a.src[q][0] / ts, by = a.src[q][1] / ts, bz = g.ndim == 3 ? a.src[q][2] / ts : 0;
        return (bz * a.nty + by) * a.ntx + bx;
    };
    if (a.list) {
        for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < a.ntiles; t += gridDim.x * blockDim.x) {
            unsigned m = 0u;
            for (int q = 0; q < a.nsrc; ++q)
                if (tile_of(q) == t) m = 1u;  // queued for iteration 0
            a.mark[t] = m;
            a.state[t] = 0u;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        unsigned n = 0;
        for (int q = 0; q < a.nsrc; ++q) {
            const int t = tile_of(q);
            bool seen = false;
            for (int p = 0; p < q; ++p) seen |= tile_of(p) == t;
            if (seen) continue;
            if (a.list) a.list[n] = t;
            else a.act[t] = 1u;
            ++n;
        }
        a.count[0] = n;
        if (a.list) {
            a.count[1] = a.count[2] = 0u;
            a.take[0] = a.take[1] = a.take[2] = 0u;
            *bar = 0u;
            for (int c = 0; c < 8; ++c) ctl->counters[c] = 0;
        }
    }
}

template <typename T>
cudaError_t launch_fim_init(const FimProblem<T>& a, int ts, int grid, cudaStream_t s, FieldCtl* ctl, unsigned* bar)
{
    fim_init_kernel<T><<<grid, 256, 0, s>>>(a, ts, ctl, bar);
    return cudaGetLastError();
}
template cudaError_t launch_fim_init<float>(const FimProblem<float>&, int, int, cudaStream_t, FieldCtl*, unsigned*);
template cudaError_t launch_fim_init<double>(const FimProblem<double>&, int, int, cudaStream_t, FieldCtl*, unsigned*);

void eik_scratch_free_impl(ripple_field f)
{
    if (!f->eik) return;
    ctx_free(f->ctx, f->eik->mem, f->eik->bytes);
    delete f->eik;
    f->eik = nullptr;
}

// Fill the problem description of a solve on (S, Tf); the caller provides the
// scratch pointers.
ripple_status fim_describe(ripple_field S, ripple_field Tf, const int64_t* src, int nsrc, double h, double tol,
                           int* ntx, int* nty, int* ntz, int* ntiles, int (*srcc)[3])
{
    const int ndim = Tf->ndim;
    const int ts = ndim == 2 ? EikTile<2>::TS : EikTile<3>::TS;
    *ntx = (Tf->geom.n[0] + ts - 1) / ts;
    *nty = (Tf->geom.n[1] + ts - 1) / ts;
    *ntz = ndim == 3 ? (Tf->geom.n[2] + ts - 1) / ts : 1;
    *ntiles = *ntx * *nty * *ntz;
    for (int q = 0; q < nsrc; ++q)
        for (int d = 0; d < 3; ++d) {
            const int64_t c = d < ndim ? src[q * ndim + d] : 0;
            if (c < 0 || c >= Tf->geom.n[d]) return fail(RIPPLE_ERR_INVALID, "source outside the grid");
            srcc[q][d] = (int)c;
        }
    (void)S;
    (void)h;
    (void)tol;
    return RIPPLE_OK;
}

}  // namespace ripple

using namespace ripple;

void eik_scratch_free(ripple_field f) { eik_scratch_free_impl(f); }

namespace ripple {
size_t fim_list_scratch_bytes(int ntiles)
{
    // count[3] + barrier + take[3] u32 (64 bytes), list[3][ntiles] i32,
    // state[ntiles] u32, mark[ntiles] u32
    return (size_t)ntiles * 5 * 4 + 64;
}

template <typename T, int DIM>
ripple_status fim_solve_lists(FimProblem<T> a, void* scratch, FieldCtl* ctl, long long max_iters, int sm_count,
                              cudaStream_t s)
{
    char* base = static_cast<char*>(scratch);
    a.count = reinterpret_cast<unsigned*>(base);
    a.take = reinterpret_cast<unsigned*>(base + 32);
    a.list = reinterpret_cast<int*>(base + 64);
    a.state = reinterpret_cast<unsigned*>(base + 64 + (size_t)a.ntiles * 3 * 4);
    a.mark = reinterpret_cast<unsigned*>(base + 64 + (size_t)a.ntiles * 4 * 4);
    a.act = nullptr;
    a.cur = nullptr;
    EikArgs e{};
    e.max_iters = max_iters > 0 ? max_iters : 1000000;
    e.bar = reinterpret_cast<unsigned*>(base + 16);
    e.spin_limit = grid_spin_limit();
    e.ctl = ctl;
    auto kern = fim_kernel<T, DIM>;
    static ResidentCtas resident;
    int per_sm = resident.get(kern, EikTile<DIM>::NT, 0);
    if (per_sm < 1) return fail(RIPPLE_ERR_INTERNAL, "FIM kernel cannot be resident");
    // 2D solves keep 100 to 300 tiles active per iteration, and an iteration
    // lasts as long as its longest visit: two CTAs per SM give most visits
    // their own issue slots (2048^2: one 1790, two 1509, four 1614 us; 1000 x 700:
    // 622, 648, 746); 3D solves have a thousand and want every resident CTA
    if (DIM == 2) per_sm = std::min(per_sm, kFimCtasPerSm2D);
    int grid = std::min(per_sm * sm_count, a.ntiles);
    grid = std::max(grid, 1);
    const long long total = (long long)a.gT.n[0] * a.gT.n[1] * a.gT.n[2];
    const int igrid = (int)std::min<long long>((total + 255) / 256, 8LL * sm_count);
    RIPPLE_CUDA(launch_fim_init<T>(a, EikTile<DIM>::TS, igrid, s, ctl, e.bar));
    void* args[] = {&a, &e};
    RIPPLE_CUDA(cudaLaunchCooperativeKernel((const void*)kern, dim3(grid), dim3(EikTile<DIM>::NT), args, 0, s));
    return RIPPLE_OK;
}
template ripple_status fim_solve_lists<float, 2>(FimProblem<float>, void*, FieldCtl*, long long, int, cudaStream_t);
template ripple_status fim_solve_lists<double, 2>(FimProblem<double>, void*, FieldCtl*, long long, int, cudaStream_t);
template ripple_status fim_solve_lists<float, 3>(FimProblem<float>, void*, FieldCtl*, long long, int, cudaStream_t);
template ripple_status fim_solve_lists<double, 3>(FimProblem<double>, void*, FieldCtl*, long long, int, cudaStream_t);
}  // namespace ripple

extern "C" ripple_status ripple_eikonal_solve(ripple_field S, ripple_field Tf, const int64_t* src, int nsrc,
                                              const ripple_eik_params* p, ripple_eik_stats* stats)
{
    if (!S || !Tf || !src || !p) return fail(RIPPLE_ERR_INVALID, "NULL argument");
    if (S->ctx != Tf->ctx) return fail(RIPPLE_ERR_INVALID, "fields of different contexts");
    if (S->ncomp != 1 || Tf->ncomp != 1) return fail(RIPPLE_ERR_INVALID, "eikonal fields have one component");
    if (S->ndim != Tf->ndim || S->dtype != Tf->dtype) return fail(RIPPLE_ERR_INVALID, "field shape/dtype mismatch");
    for (int d = 0; d < 3; ++d)
        if (S->geom.n[d] != Tf->geom.n[d]) return fail(RIPPLE_ERR_INVALID, "field dims differ");
    if (nsrc < 1 || nsrc > kMaxSources) return fail(RIPPLE_ERR_INVALID, "need 1..16 sources");
    if (!(p->h > 0.0) || !(p->tol > 0.0)) return fail(RIPPLE_ERR_INVALID, "need h > 0 and tol > 0");
    const int ndim = Tf->ndim;
    int ntx, nty, ntz, ntiles;
    int srcc[kMaxSources][3];
    ripple_status st = fim_describe(S, Tf, src, nsrc, p->h, p->tol, &ntx, &nty, &ntz, &ntiles, srcc);
    if (st != RIPPLE_OK) return st;
    ripple_ctx ctx = Tf->ctx;
    st = ensure_second_buffer(Tf);
    if (st != RIPPLE_OK) return st;
    const size_t need = fim_list_scratch_bytes(ntiles);
    if (!Tf->eik || Tf->eik->bytes < need) {
        eik_scratch_free(Tf);
        Tf->eik = new EikScratch();
        st = ctx_alloc(ctx, need, &Tf->eik->mem);
        if (st != RIPPLE_OK) {
            delete Tf->eik;
            Tf->eik = nullptr;
            return st;
        }
        Tf->eik->bytes = need;
        Tf->eik->ntiles = ntiles;
    }
    cudaStream_t s = ctx->stream;
    const long long max_iters = p->max_iters > 0 ? p->max_iters : 1000000;
    auto fill = [&](auto& a) {
        using TT = std::remove_pointer_t<decltype(a.slow)>;
        using TV = std::remove_const_t<TT>;
        a.buf[0] = static_cast<TV*>(Tf->buf[0]);
        a.buf[1] = static_cast<TV*>(Tf->buf[1]);
        a.slow = static_cast<const TV*>(S->buf[S->cur]);
        a.gT = Tf->geom;
        a.gS = S->geom;
        a.ntx = ntx; a.nty = nty; a.ntz = ntz; a.ntiles = ntiles;
        a.nsrc = nsrc;
        for (int q = 0; q < nsrc; ++q)
            for (int d = 0; d < 3; ++d) a.src[q][d] = srcc[q][d];
        a.h = p->h;
        a.tol = p->tol;
    };
    void* mem = Tf->eik->mem;
    if (Tf->dtype == RIPPLE_F32) {
        FimProblem<float> a{};
        fill(a);
        st = ndim == 2 ? fim_solve_lists<float, 2>(a, mem, Tf->ctl, max_iters, ctx->sm_count, s)
                       : fim_solve_lists<float, 3>(a, mem, Tf->ctl, max_iters, ctx->sm_count, s);
    } else {
        FimProblem<double> a{};
        fill(a);
        st = ndim == 2 ? fim_solve_lists<double, 2>(a, mem, Tf->ctl, max_iters, ctx->sm_count, s)
                       : fim_solve_lists<double, 3>(a, mem, Tf->ctl, max_iters, ctx->sm_count, s);
    }
    if (st != RIPPLE_OK) return st;
    Tf->cur = 0;
    RIPPLE_CUDA(cudaMemcpyAsync(ctx->h_ctl, Tf->ctl, sizeof(FieldCtl), cudaMemcpyDeviceToHost, s));
    RIPPLE_CUDA(cudaStreamSynchronize(s));
    const FieldCtl host = *ctx->h_ctl;
    if (stats) {
        stats->iterations = host.counters[0];
        stats->tile_visits = host.counters[1];
        stats->cell_updates = host.counters[2];
    }
    if (host.err) {
        RIPPLE_CUDA(cudaMemsetAsync(&Tf->ctl->err, 0, sizeof(unsigned), s));
        if (host.err & DEV_ERR_BARRIER)
            return fail(RIPPLE_ERR_TIMEOUT, "FIM grid barrier wait ran out (a CTA was not resident or stalled)");
        if (host.err & DEV_ERR_TIMEOUT) return fail(RIPPLE_ERR_TIMEOUT, "FIM did not converge within max_iters");
        return fail(RIPPLE_ERR_INTERNAL, "FIM device error");
    }
    return RIPPLE_OK;
}
