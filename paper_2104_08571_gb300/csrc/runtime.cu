// C-ABI runtime: contexts, fields, tensor maps, upload/download and the
// Euler step driver.  No kernel arithmetic lives here.
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>

#include "grid_sync.cuh"
#include "runtime.h"
#include "step_budget.h"

namespace ripple {

static thread_local std::string g_last_error;

void set_error(const std::string& msg) { g_last_error = msg; }

ripple_status fail(ripple_status st, const std::string& msg)
{
    set_error(msg);
    return st;
}

ripple_status cuda_fail(cudaError_t e, const char* what)
{
    set_error(std::string(what) + ": " + cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? RIPPLE_ERR_OOM : RIPPLE_ERR_CUDA;
}

size_t elem_size(ripple_dtype d) { return d == RIPPLE_F64 ? 8 : 4; }

static size_t round_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

bool budget_reserve(ripple_ctx ctx, size_t bytes)
{
    size_t cur = ctx->used.load();
    for (;;) {
        if (ctx->budget && cur + bytes > ctx->budget) return false;
        if (ctx->used.compare_exchange_weak(cur, cur + bytes)) return true;
    }
}

FieldGeom make_field_geom(int ndim, const int64_t* dims, int ncomp, ripple_layout layout, int halo,
                          ripple_dtype dtype, size_t* bytes)
{
    const int es = (int)elem_size(dtype);
    const int a = 16 / es;  // 16-byte x alignment in cells
    FieldGeom g{};
    g.ndim = ndim;
    g.ncomp = ncomp;
    g.h = halo;
    g.lead = (a - halo % a) % a;
    for (int d = 0; d < 3; ++d) g.n[d] = d < ndim ? (int)dims[d] : 1;
    g.px = (long long)round_up((size_t)(g.lead + g.n[0] + 2 * halo), (size_t)a);
    g.py = g.n[1] + 2 * halo;
    g.pz = ndim == 3 ? g.n[2] + 2 * halo : 1;
    const long long ncell = g.px * g.py * g.pz;
    if (layout == RIPPLE_SOA) {
        g.cell_stride = 1;
        g.comp_stride = ncell;
    } else {
        g.cell_stride = ncomp;
        g.comp_stride = 1;
    }
    if (bytes) *bytes = round_up((size_t)ncell * ncomp * es, 256);
    return g;
}

bool fault_injected(const char* step)
{
    const char* env = std::getenv("RIPPLE_FAULT");
    if (!env || !*env) return false;
    const size_t n = std::strlen(step);
    for (const char* p = env; *p;) {
        const char* e = std::strchr(p, ',');
        const size_t len = e ? (size_t)(e - p) : std::strlen(p);
        if (len == n && std::strncmp(p, step, n) == 0) return true;
        if (!e) break;
        p = e + 1;
    }
    return false;
}

ripple_status ctx_alloc(ripple_ctx ctx, size_t bytes, void** out)
{
    *out = nullptr;
    if (fault_injected("alloc")) return fail(RIPPLE_ERR_OOM, "device allocation failed (injected: RIPPLE_FAULT=alloc)");
    bytes = round_up(std::max<size_t>(bytes, 256), 256);
    if (!budget_reserve(ctx, bytes))
        return fail(RIPPLE_ERR_BUDGET, "allocation of " + std::to_string(bytes) + " bytes exceeds the memory budget");
    void* p = nullptr;
    if (ctx->alloc_fn) {
        p = ctx->alloc_fn(bytes, ctx->alloc_user);
        if (!p) {
            ctx->used -= bytes;
            return fail(RIPPLE_ERR_OOM, "allocator callback returned NULL");
        }
        if (reinterpret_cast<uintptr_t>(p) % 256) {
            ctx->free_fn(p, ctx->alloc_user);
            ctx->used -= bytes;
            return fail(RIPPLE_ERR_INTERNAL, "allocator callback returned memory not aligned to 256 bytes");
        }
    } else {
        cudaError_t e = cudaMalloc(&p, bytes);
        if (e != cudaSuccess) {
            ctx->used -= bytes;
            return cuda_fail(e, "cudaMalloc");
        }
    }
    *out = p;
    return RIPPLE_OK;
}

void ctx_free(ripple_ctx ctx, void* p, size_t bytes)
{
    if (!p) return;
    bytes = round_up(std::max<size_t>(bytes, 256), 256);
    if (ctx->alloc_fn) ctx->free_fn(p, ctx->alloc_user);
    else cudaFree(p);
    ctx->used -= bytes;
}

static PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

ripple_status encode_plane_map(void* buffer, const FieldGeom& g, ripple_layout layout, ripple_dtype dtype, int kind,
                               int r, int tx, int ty, CUtensorMap* out)
{
    auto enc = encode_fn();
    if (!enc) return fail(RIPPLE_ERR_CUDA, "cuTensorMapEncodeTiled is unavailable");
    const int es = (int)elem_size(dtype);
    const int nc = g.ncomp;
    const bool soa = layout == RIPPLE_SOA;
    cuuint64_t dims[4], strides[3];
    cuuint32_t box[4], estr[4] = {1, 1, 1, 1};
    cuuint32_t rank;
    char* base = static_cast<char*>(buffer);
    const BoxGeom bg = plane_box(es, nc, !soa, r, tx, ty);
    if (kind == 2) {
        // AoS plane staging of the row kernel: each row viewed as groups of
        // four cells (4 x ncomp elements, a multiple of 16 bytes), so a box
        // as wide as the row tile fits the 256-element box limit per dimension
        if (soa || g.ndim != 3 || g.px % 4 != 0 || bg.bx % 4 != 0)
            return fail(RIPPLE_ERR_INTERNAL, "grouped AoS plane map needs a 3D AoS field");
        rank = 4;
        dims[0] = 4 * nc; dims[1] = g.px / 4; dims[2] = g.py; dims[3] = g.pz;
        strides[0] = 4 * nc * es; strides[1] = g.px * nc * es; strides[2] = g.px * nc * g.py * es;
        box[0] = 4 * nc; box[1] = bg.bx / 4; box[2] = bg.by; box[3] = 1;
    } else if (kind == 0) {
        if (soa) {
            dims[0] = g.px; dims[1] = g.py;
            strides[0] = g.px * es; strides[1] = g.px * g.py * es;
            box[0] = bg.bx; box[1] = bg.by;
            if (g.ndim == 3) {
                rank = 4;
                dims[2] = g.pz; dims[3] = nc;
                strides[2] = g.px * g.py * g.pz * es;
                box[2] = 1; box[3] = nc;
            } else {
                rank = 3;
                dims[2] = nc;
                box[2] = nc;
            }
        } else {
            dims[0] = g.px * nc; dims[1] = g.py;
            strides[0] = g.px * nc * es;
            box[0] = bg.bx * nc; box[1] = bg.by;
            if (g.ndim == 3) {
                rank = 3;
                dims[2] = g.pz;
                strides[1] = g.px * nc * g.py * es;
                box[2] = 1;
            } else {
                rank = 2;
            }
        }
    } else {
        base += geom_elem(g, 0, 0, 0, 0) * es;
        if (soa) {
            dims[0] = g.n[0]; dims[1] = g.n[1];
            strides[0] = g.px * es; strides[1] = g.px * g.py * es;
            box[0] = tx; box[1] = ty;
            if (g.ndim == 3) {
                rank = 4;
                dims[2] = g.n[2]; dims[3] = nc;
                strides[2] = g.px * g.py * g.pz * es;
                box[2] = 1; box[3] = nc;
            } else {
                rank = 3;
                dims[2] = nc;
                box[2] = nc;
            }
        } else {
            dims[0] = (cuuint64_t)g.n[0] * nc; dims[1] = g.n[1];
            strides[0] = g.px * nc * es;
            box[0] = tx * nc; box[1] = ty;
            if (g.ndim == 3) {
                rank = 3;
                dims[2] = g.n[2];
                strides[1] = g.px * nc * g.py * es;
                box[2] = 1;
            } else {
                rank = 2;
            }
        }
    }
    CUresult cr = enc(out, dtype == RIPPLE_F64 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32,
                      rank, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                      CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                      // staging loads read NaN beyond the tensor (as the padded cells of an Euler
                      // field); stores are clipped and fill nothing
                      kind != 1 ? CU_TENSOR_MAP_FLOAT_OOB_FILL_NAN_REQUEST_ZERO_FMA : CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (cr != CUDA_SUCCESS)
        return fail(RIPPLE_ERR_CUDA, "cuTensorMapEncodeTiled failed (code " + std::to_string((int)cr) + ")");
    return RIPPLE_OK;
}

const CUtensorMap* field_map(ripple_field f, int buffer, int kind, int r, int tx, int ty, ripple_status* st)
{
    *st = RIPPLE_OK;
    for (auto& m : f->maps)
        if (m.buffer == buffer && m.kind == kind && m.r == r && m.tx == tx && m.ty == ty) return &m.map;
    MapEntry e{};
    e.buffer = buffer; e.kind = kind; e.r = r; e.tx = tx; e.ty = ty;
    *st = encode_plane_map(f->buf[buffer], f->geom, f->layout, f->dtype, kind, r, tx, ty, &e.map);
    if (*st != RIPPLE_OK) return nullptr;
    f->maps.push_back(e);
    return &f->maps.back().map;
}

ripple_status ensure_second_buffer(ripple_field f)
{
    if (f->buf[1]) return RIPPLE_OK;
    void* p = nullptr;
    ripple_status st = ctx_alloc(f->ctx, f->bytes, &p);
    if (st != RIPPLE_OK) return st;
    f->buf[1] = p;  // every cell is written before it is read (Euler padding: pad_fill_nan_kernel)
    f->maps.clear();  // vector may reallocate: entries are re-encoded on demand
    return RIPPLE_OK;
}

static ripple_status map_dev_err(unsigned err, const FieldCtl* host = nullptr)
{
    if (err & DEV_ERR_INTERNAL) return fail(RIPPLE_ERR_INTERNAL, "device-side invariant violated");
    if (err & DEV_ERR_BARRIER) return fail(RIPPLE_ERR_TIMEOUT, "a device-side grid barrier wait ran out");
    if (err & DEV_ERR_TIMEOUT) return fail(RIPPLE_ERR_TIMEOUT, "a device-side bounded wait ran out");
    if (err & DEV_ERR_NUMERIC) {
        std::string msg = "non-positive or NaN density/pressure produced";
        if (host && host->counters[4] > 0) {
            const long long c = host->counters[4];
            const char* what = c == BAD_CELL    ? "updated cell"
                               : c == BAD_INPUT ? "input cell"
                                                : "reconstructed/predicted/face state in the tile starting at cell";
            msg += std::string(" (first at ") + what + " (" + std::to_string(host->counters[5]) + ", " +
                   std::to_string(host->counters[6]) + ", " + std::to_string(host->counters[7]) + "))";
        }
        return fail(RIPPLE_ERR_NUMERIC, msg);
    }
    return RIPPLE_OK;
}

ripple_status take_device_error(ripple_field f)
{
    FieldCtl* h = f->ctx->h_ctl;
    RIPPLE_CUDA(cudaMemcpyAsync(&h->err, &f->ctl->err, sizeof(unsigned), cudaMemcpyDeviceToHost, f->ctx->stream));
    RIPPLE_CUDA(cudaStreamSynchronize(f->ctx->stream));
    const unsigned err = h->err;
    if (err) RIPPLE_CUDA(cudaMemsetAsync(&f->ctl->err, 0, sizeof(unsigned), f->ctx->stream));
    return map_dev_err(err);
}

// Euler step dispatch -------------------------------------------------------

cudaError_t sweep_launch(ripple_dtype dt, int dim, int layout, int scheme, int v, const SweepLaunch& L)
{
    if (dt == RIPPLE_F32) return dim == 2 ? sweep_launch_f32_2d(layout, scheme, v, L) : sweep_launch_f32_3d(layout, scheme, v, L);
    return dim == 2 ? sweep_launch_f64_2d(layout, scheme, v, L) : sweep_launch_f64_3d(layout, scheme, v, L);
}
int sweep_smem(ripple_dtype dt, int dim, int layout, int scheme, int v)
{
    if (dt == RIPPLE_F32) return dim == 2 ? sweep_smem_f32_2d(layout, scheme, v) : sweep_smem_f32_3d(layout, scheme, v);
    return dim == 2 ? sweep_smem_f64_2d(layout, scheme, v) : sweep_smem_f64_3d(layout, scheme, v);
}
int sweep_occ(ripple_dtype dt, int dim, int layout, int scheme, int v)
{
    if (dt == RIPPLE_F32) return dim == 2 ? sweep_occ_f32_2d(layout, scheme, v) : sweep_occ_f32_3d(layout, scheme, v);
    return dim == 2 ? sweep_occ_f64_2d(layout, scheme, v) : sweep_occ_f64_3d(layout, scheme, v);
}

// Rows per walk for `lines` independent lines of n rows on `sms` SMs of 16
// resident warps, a walk of R rows costing R + extra.  In units of the time a
// warp alone takes for a row, a scheduler with enough warps finishes a row
// every 0.28 (a warp issues about every fourth cycle).  Walks that all have a
// warp of their own end together; otherwise the last one handed out ends about
// 0.6 walks after the schedulers have run out of others.  `most` bounds R:
// walks along z keep as many planes in flight as they are long and lose L2
// hits (200 x 171 x 186: 8 planes 149 us a step, 31 190, 62 223), and long
// in-plane walks of a 3D field do the same (24 rows).
static void walk_split(long long lines, int n, int sms, double extra, int most, int* rows, int* segs)
{
    double best = 1e300;
    *rows = n;
    *segs = 1;
    for (int r = 1; r <= std::min(n, most); ++r) {
        const int sg = (n + r - 1) / r;
        const long long units = lines * sg, per = (units + 4 * sms - 1) / (4 * sms);  // walks per scheduler
        const double cost = units <= (long long)kWalkWarps * sms
                                ? (r + extra) * std::max(1.0, 0.28 * (double)per)
                                : (r + extra) * ((double)units * 0.28 / (4.0 * sms) + 0.6);
        if (cost < best) {
            best = cost;
            *rows = r;
            *segs = sg;
        }
    }
}

// Geometry, parameters and work split of a walk launch; returns its grid.
static int walk_plan(const ripple_ctx_s* ctx, WalkStep& a, const FieldGeom& g, bool f64, int scheme, double gamma,
                     double cfl, const double* dx, int bc, int occ)
{
    const bool d3 = g.ndim == 3;
    const int sms = ctx->sm_count;
    a.g = g;
    a.cfl = cfl;
    a.gamma = gamma;
    a.gamma_f = (float)gamma;
    a.gm1_f = (float)(gamma - 1.0);
    for (int d = 0; d < g.ndim; ++d) {
        a.inv_dx[d] = 1.0 / dx[d];
        a.dx_cfl[d] = dx[d] / cfl;
        a.inv_dx_f[d] = (float)a.inv_dx[d];
    }
    a.bc = bc;
    a.spin_limit = grid_spin_limit();
    if (f64) {
        tile64_plan(a, sms);
        return (int)std::min<long long>((long long)occ * sms, (long long)a.strips * a.segs);
    }
    a.strips = (g.n[0] + kWalkUse - 1) / kWalkUse;
    walk_split((long long)a.strips * g.n[2], g.n[1], sms, scheme == SCHEME_RUSANOV1 ? 1.5 : 2.0, d3 ? 24 : 128, &a.rows,
               &a.segs);
    // unit numbers are 32-bit: at most 2^32 padded cells, and a row (at least 8 of them) gives a unit per 60 columns
    long long units = (long long)a.strips * a.segs * g.n[2];
    if (d3) {
        a.zstrips = (g.n[0] + 63) / 64;
        walk_split((long long)a.zstrips * g.n[1], g.n[2], sms, 1.0, 8, &a.zrows, &a.zsegs);
        units = std::max(units, (long long)a.zstrips * g.n[1] * a.zsegs);
    }
    return (int)std::min<long long>((long long)occ * sms, units);
}

cudaError_t walk2d_solo_launch(ripple_ctx ctx, WalkStep& a, const FieldGeom& g, const ripple_fv_params& p,
                               ripple_layout layout, cudaStream_t s)
{
    const int lay = layout == RIPPLE_SOA ? LAYOUT_SOA : LAYOUT_AOS;
    const int occ = walk2d_occ_f32(SCHEME_RUSANOV1, lay);
    if (occ <= 0) return cudaErrorInvalidValue;
    const int grid = walk_plan(ctx, a, g, false, SCHEME_RUSANOV1, p.gamma, p.cfl, p.dx, (int)p.bc, occ);
    return walk2d_launch_f32(SCHEME_RUSANOV1, lay, a, grid, s);
}

}  // namespace ripple

using namespace ripple;

extern "C" {

const char* ripple_last_error(void) { return g_last_error.c_str(); }

const char* ripple_version(void) { return "ripple-gb300 0.1 (sm_103a)"; }

ripple_status ripple_ctx_create(int device, size_t mem_budget_bytes, ripple_ctx* out)
{
    if (!out) return fail(RIPPLE_ERR_INVALID, "out is NULL");
    *out = nullptr;
    int n = 0;
    RIPPLE_CUDA(cudaGetDeviceCount(&n));
    if (device < 0 || device >= n) return fail(RIPPLE_ERR_INVALID, "no such CUDA device");
    RIPPLE_CUDA(cudaSetDevice(device));
    auto* c = new (std::nothrow) ripple_ctx_s();
    if (!c) return fail(RIPPLE_ERR_OOM, "host allocation failed");
    c->device = device;
    c->budget = mem_budget_bytes;
    cudaError_t e = cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, device);
    if (e == cudaSuccess) e = cudaMallocHost(reinterpret_cast<void**>(&c->h_ctl), sizeof(FieldCtl));
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&c->own_stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) {
        if (c->h_ctl) cudaFreeHost(c->h_ctl);
        delete c;
        return cuda_fail(e, "ripple_ctx_create");
    }
    c->stream = c->own_stream;
    *out = c;
    return RIPPLE_OK;
}

ripple_status ripple_ctx_destroy(ripple_ctx ctx)
{
    if (!ctx) return RIPPLE_OK;
    if (ctx->nfields.load() != 0) return fail(RIPPLE_ERR_INVALID, "destroy all fields before their context");
    batch_runtime_destroy(ctx);
    cudaStreamSynchronize(ctx->stream);
    ctx_free(ctx, ctx->staging, ctx->staging_bytes);
    ctx_free(ctx, ctx->partials, ctx->partials_bytes);
    if (ctx->own_stream) cudaStreamDestroy(ctx->own_stream);
    cudaFreeHost(ctx->h_ctl);
    delete ctx;
    return RIPPLE_OK;
}

ripple_status ripple_set_stream(ripple_ctx ctx, void* cuda_stream)
{
    if (!ctx) return fail(RIPPLE_ERR_INVALID, "ctx is NULL");
    ctx->stream = cuda_stream ? static_cast<cudaStream_t>(cuda_stream) : ctx->own_stream;
    return RIPPLE_OK;
}

ripple_status ripple_set_allocator(ripple_ctx ctx, void* (*alloc)(size_t, void*), void (*release)(void*, void*),
                                   void* user)
{
    if (!ctx) return fail(RIPPLE_ERR_INVALID, "ctx is NULL");
    if (ctx->used.load() != 0) return fail(RIPPLE_ERR_INVALID, "set the allocator before allocating");
    if ((alloc == nullptr) != (release == nullptr)) return fail(RIPPLE_ERR_INVALID, "alloc and release go together");
    ctx->alloc_fn = alloc;
    ctx->free_fn = release;
    ctx->alloc_user = user;
    return RIPPLE_OK;
}

ripple_status ripple_ctx_sync(ripple_ctx ctx)
{
    if (!ctx) return fail(RIPPLE_ERR_INVALID, "ctx is NULL");
    RIPPLE_CUDA(cudaStreamSynchronize(ctx->stream));
    std::vector<ripple_field> fields;
    {
        std::lock_guard<std::mutex> lk(ctx->mu);
        fields = ctx->fields;
    }
    ripple_status first = RIPPLE_OK;
    for (ripple_field f : fields) {
        ripple_status st = take_device_error(f);
        if (first == RIPPLE_OK) first = st;
    }
    if (layout_bench_take_error(ctx->stream) && first == RIPPLE_OK)
        first = fail(RIPPLE_ERR_TIMEOUT, "a bounded wait of a staged particle update ran out");
    return first;
}

ripple_status ripple_ctx_mem_used(ripple_ctx ctx, size_t* bytes)
{
    if (!ctx || !bytes) return fail(RIPPLE_ERR_INVALID, "NULL argument");
    *bytes = ctx->used.load();
    return RIPPLE_OK;
}

ripple_status ripple_field_create(ripple_ctx ctx, int ndim, const int64_t* dims, int ncomp, ripple_layout layout,
                                  int halo, ripple_dtype dtype, ripple_field* out)
{
    if (!out) return fail(RIPPLE_ERR_INVALID, "out is NULL");
    *out = nullptr;
    if (!ctx || !dims) return fail(RIPPLE_ERR_INVALID, "NULL argument");
    if (ndim < 2 || ndim > 3) return fail(RIPPLE_ERR_INVALID, "ndim must be 2 or 3");
    if (ncomp < 1 || ncomp > 5) return fail(RIPPLE_ERR_INVALID, "ncomp must be 1..5");
    if (halo < 0 || halo > 8) return fail(RIPPLE_ERR_INVALID, "halo must be 0..8");
    if (layout != RIPPLE_AOS && layout != RIPPLE_SOA) return fail(RIPPLE_ERR_INVALID, "bad layout");
    if (dtype != RIPPLE_F32 && dtype != RIPPLE_F64) return fail(RIPPLE_ERR_INVALID, "bad dtype");
    for (int d = 0; d < ndim; ++d)
        if (dims[d] < 1 || dims[d] > (1 << 20)) return fail(RIPPLE_ERR_INVALID, "dims out of range");
    auto* f = new (std::nothrow) ripple_field_s();
    if (!f) return fail(RIPPLE_ERR_OOM, "host allocation failed");
    f->ctx = ctx;
    f->ndim = ndim;
    f->ncomp = ncomp;
    f->halo = halo;
    f->layout = layout;
    f->dtype = dtype;
    f->geom = make_field_geom(ndim, dims, ncomp, layout, halo, dtype, &f->bytes);
    const FieldGeom& g = f->geom;
    // at most 2^32 padded cells per buffer: byte counts stay far from overflow
    // and every tile, item and table count of the kernels fits in 32 bits
    if (g.px * g.py * g.pz > (1LL << 32)) {
        delete f;
        return fail(RIPPLE_ERR_INVALID, "field too large: more than 2^32 padded cells per buffer");
    }
    f->elems = (size_t)(g.px * g.py * g.pz) * ncomp;
    ripple_status st = ctx_alloc(ctx, f->bytes, &f->buf[0]);
    if (st == RIPPLE_OK) st = ctx_alloc(ctx, sizeof(FieldCtl), reinterpret_cast<void**>(&f->ctl));
    if (st != RIPPLE_OK) {
        ctx_free(ctx, f->buf[0], f->bytes);
        delete f;
        return st;
    }
    cudaError_t e = cudaMemsetAsync(f->buf[0], 0, f->bytes, ctx->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(f->ctl, 0, sizeof(FieldCtl), ctx->stream);
    if (e != cudaSuccess) {
        ctx_free(ctx, f->buf[0], f->bytes);
        ctx_free(ctx, f->ctl, sizeof(FieldCtl));
        delete f;
        return cuda_fail(e, "cudaMemsetAsync");
    }
    ctx->nfields++;
    {
        std::lock_guard<std::mutex> lk(ctx->mu);
        ctx->fields.push_back(f);
    }
    *out = f;
    return RIPPLE_OK;
}

ripple_status ripple_field_destroy(ripple_field f)
{
    if (!f) return RIPPLE_OK;
    ripple_ctx ctx = f->ctx;
    cudaStreamSynchronize(ctx->stream);
    eik_scratch_free(f);
    ctx_free(ctx, f->buf[0], f->bytes);
    ctx_free(ctx, f->buf[1], f->bytes);
    ctx_free(ctx, f->ctl, sizeof(FieldCtl));
    ctx->nfields--;
    {
        std::lock_guard<std::mutex> lk(ctx->mu);
        ctx->fields.erase(std::remove(ctx->fields.begin(), ctx->fields.end(), f), ctx->fields.end());
    }
    delete f;
    return RIPPLE_OK;
}

static ripple_status ensure_staging(ripple_ctx ctx, size_t bytes)
{
    if (ctx->staging_bytes >= bytes) return RIPPLE_OK;
    RIPPLE_CUDA(cudaStreamSynchronize(ctx->stream));
    ctx_free(ctx, ctx->staging, ctx->staging_bytes);
    ctx->staging = nullptr;
    ctx->staging_bytes = 0;
    ripple_status st = ctx_alloc(ctx, bytes, &ctx->staging);
    if (st != RIPPLE_OK) return st;
    ctx->staging_bytes = round_up(bytes, 256);
    return RIPPLE_OK;
}

static size_t interior_bytes(ripple_field f)
{
    const FieldGeom& g = f->geom;
    return (size_t)g.n[0] * g.n[1] * g.n[2] * f->ncomp * elem_size(f->dtype);
}

ripple_status ripple_field_upload_device(ripple_field f, const void* src, ripple_layout src_layout)
{
    if (!f || !src) return fail(RIPPLE_ERR_INVALID, "NULL argument");
    if (src_layout != RIPPLE_AOS && src_layout != RIPPLE_SOA) return fail(RIPPLE_ERR_INVALID, "bad layout");
    RIPPLE_CUDA(launch_interior_copy(f->dtype, f->buf[f->cur], f->geom, const_cast<void*>(src), src_layout, 0,
                                     8 * f->ctx->sm_count, f->ctx->stream));
    f->prepared = false;
    return RIPPLE_OK;
}

ripple_status ripple_field_download_device(ripple_field f, void* dst, ripple_layout dst_layout)
{
    if (!f || !dst) return fail(RIPPLE_ERR_INVALID, "NULL argument");
    if (dst_layout != RIPPLE_AOS && dst_layout != RIPPLE_SOA) return fail(RIPPLE_ERR_INVALID, "bad layout");
    RIPPLE_CUDA(launch_interior_copy(f->dtype, f->buf[f->cur], f->geom, dst, dst_layout, 1, 8 * f->ctx->sm_count,
                                     f->ctx->stream));
    return RIPPLE_OK;
}

ripple_status ripple_field_upload(ripple_field f, const void* src, ripple_layout src_layout)
{
    if (!f || !src) return fail(RIPPLE_ERR_INVALID, "NULL argument");
    const size_t bytes = interior_bytes(f);
    ripple_status st = ensure_staging(f->ctx, bytes);
    if (st != RIPPLE_OK) return st;
    RIPPLE_CUDA(cudaMemcpyAsync(f->ctx->staging, src, bytes, cudaMemcpyHostToDevice, f->ctx->stream));
    st = ripple_field_upload_device(f, f->ctx->staging, src_layout);
    if (st != RIPPLE_OK) return st;
    RIPPLE_CUDA(cudaStreamSynchronize(f->ctx->stream));
    return RIPPLE_OK;
}

ripple_status ripple_field_download(ripple_field f, void* dst, ripple_layout dst_layout)
{
    if (!f || !dst) return fail(RIPPLE_ERR_INVALID, "NULL argument");
    const size_t bytes = interior_bytes(f);
    ripple_status st = ensure_staging(f->ctx, bytes);
    if (st != RIPPLE_OK) return st;
    st = ripple_field_download_device(f, f->ctx->staging, dst_layout);
    if (st != RIPPLE_OK) return st;
    RIPPLE_CUDA(cudaMemcpyAsync(dst, f->ctx->staging, bytes, cudaMemcpyDeviceToHost, f->ctx->stream));
    return take_device_error(f);
}

ripple_status ripple_field_describe(ripple_field f, ripple_field_desc* out)
{
    if (!f || !out) return fail(RIPPLE_ERR_INVALID, "NULL argument");
    const FieldGeom& g = f->geom;
    out->ndim = f->ndim;
    out->ncomp = f->ncomp;
    out->halo = f->halo;
    out->layout = f->layout;
    out->dtype = f->dtype;
    for (int d = 0; d < 3; ++d) out->dims[d] = g.n[d];
    out->padded[0] = g.px;
    out->padded[1] = g.py;
    out->padded[2] = g.pz;
    out->x_lead = g.lead;
    out->buffer_bytes = f->bytes;
    out->current = f->buf[f->cur];
    return RIPPLE_OK;
}

ripple_status ripple_field_set_sweep(ripple_field f, int variant, int zchunk)
{
    if (!f) return fail(RIPPLE_ERR_INVALID, "NULL field");
    if (variant < -1 || variant >= kNumSweepVariants) return fail(RIPPLE_ERR_INVALID, "unknown sweep variant");
    if (zchunk < 0) return fail(RIPPLE_ERR_INVALID, "zchunk must be >= 0");
    f->variant = variant;
    f->zchunk = zchunk;
    return RIPPLE_OK;
}

// Steps of a field by the multi-step kernels: FP32 strip walks (every 2D
// scheme, and the split FORCE step in 3D) and the FP64 first-order 2D tiles.
static ripple_status walk_field_steps(ripple_field U, const ripple_fv_params& p, int scheme, int layout, int64_t nsteps)
{
    ripple_ctx ctx = U->ctx;
    const FieldGeom& g = U->geom;
    const bool force = scheme == SCHEME_FORCE;
    const bool d3 = U->ndim == 3;  // FORCE only
    const bool f64 = U->dtype == RIPPLE_F64;  // first-order 2D only
    const int occ = f64     ? tile64_occ()
                    : d3      ? force_walk_occ_f32_3d(layout)
                    : force ? force_walk_occ_f32_2d(layout)
                            : walk2d_occ_f32(scheme, layout);
    if (occ <= 0) return fail(RIPPLE_ERR_INTERNAL, "walk kernel does not fit");
    WalkStep a{};
    for (int b = 0; b < 2; ++b) a.buf[b] = static_cast<float*>(U->buf[b]);
    a.ctl = U->ctl;
    a.err = &U->ctl->err;
    const int grid = walk_plan(ctx, a, g, f64, scheme, p.gamma, p.cfl, p.dx, (int)p.bc, occ);
    for (int64_t done = 0; done < nsteps;) {
        a.K = walk_steps(f64, (long long)g.n[0] * g.n[1] * g.n[2], nsteps - done);
        a.cur = U->cur;
        a.slot = (int)(U->steps_total % 3);
        a.first = done == 0;
        RIPPLE_CUDA(f64     ? tile64_launch(a, grid, ctx->stream)
                    : d3    ? force_walk_launch_f32_3d(layout, a, grid, ctx->stream)
                    : force ? force_walk_launch_f32_2d(layout, a, grid, ctx->stream)
                            : walk2d_launch_f32(scheme, layout, a, grid, ctx->stream));
        if (!d3) U->cur = (U->cur + a.K) & 1;  // 3D: the z walks bring the state back
        U->steps_total += a.K;
        done += a.K;
    }
    return RIPPLE_OK;
}

ripple_status ripple_fv_step(ripple_field U, const ripple_fv_params* p, int64_t nsteps, ripple_fv_stats* stats)
{
    if (!U || !p) return fail(RIPPLE_ERR_INVALID, "NULL argument");
    if (nsteps < 0) return fail(RIPPLE_ERR_INVALID, "nsteps < 0");
    if (U->ncomp != U->ndim + 2) return fail(RIPPLE_ERR_INVALID, "Euler fields need ncomp = ndim + 2");
    if (p->scheme != RIPPLE_RUSANOV1 && p->scheme != RIPPLE_MUSCL_HANCOCK_MINMOD && p->scheme != RIPPLE_FORCE_SPLIT)
        return fail(RIPPLE_ERR_INVALID, "bad scheme");
    if (p->bc != RIPPLE_BC_PERIODIC && p->bc != RIPPLE_BC_TRANSMISSIVE) return fail(RIPPLE_ERR_INVALID, "bad bc");
    const int R = p->scheme == RIPPLE_MUSCL_HANCOCK_MINMOD ? 2 : 1;
    if (U->halo < R) return fail(RIPPLE_ERR_INVALID, "halo smaller than the stencil radius");
    if (!(p->gamma > 1.0) || !(p->cfl > 0.0)) return fail(RIPPLE_ERR_INVALID, "need gamma > 1 and cfl > 0");
    const FieldGeom& g = U->geom;
    for (int d = 0; d < U->ndim; ++d) {
        if (!(p->dx[d] > 0.0)) return fail(RIPPLE_ERR_INVALID, "dx must be > 0");
        if (p->bc == RIPPLE_BC_PERIODIC && g.n[d] < U->halo)
            return fail(RIPPLE_ERR_INVALID, "periodic axes need at least halo cells");
    }
    ripple_ctx ctx = U->ctx;
    ripple_status st = ensure_second_buffer(U);
    if (st != RIPPLE_OK) return st;
    if (!U->pad_nan) {
        // stencil items beyond the ghost layers then read NaN (ignored by the
        // admissibility minimum); prep below refills the current face ghosts
        RIPPLE_CUDA(launch_pad_nan(U->dtype, U->buf[0], U->buf[1], g, 8 * ctx->sm_count, ctx->stream));
        U->pad_nan = true;
        U->prepared = false;
    }

    const int layout = U->layout == RIPPLE_SOA ? LAYOUT_SOA : LAYOUT_AOS;
    const int scheme = p->scheme == RIPPLE_MUSCL_HANCOCK_MINMOD ? SCHEME_MUSCL
                       : p->scheme == RIPPLE_FORCE_SPLIT    ? SCHEME_FORCE
                                                            : SCHEME_RUSANOV1;
    const bool split = scheme == SCHEME_FORCE;
    // Planes per z work item of variant c: items run in rounds of the resident
    // CTAs, each costing its planes plus about one (pipeline fill, the z states
    // below its first plane), so the chunk with the fewest plane times over all
    // rounds, up to 16 planes: longer ones spread the planes in flight over
    // more of the field and lose L2 hits (256^3: 16 planes 499 us a step, 33 536,
    // 66 568).  A fixed 32 left most SMs idle on small grids (48^3
    // MUSCL-Hancock: 8 items on 152 SMs, 146 us a step; 2 planes per item 15 us).
    auto z_split = [&](int c, int* chunk) -> double {
        const long long tiles = (long long)((g.n[0] + kSweepVariants[c].tx - 1) / kSweepVariants[c].tx) *
                                ((g.n[1] + kSweepVariants[c].ty - 1) / kSweepVariants[c].ty);
        const long long slots = (long long)std::max(1, sweep_occ(U->dtype, U->ndim, layout, scheme, c)) * ctx->sm_count;
        double best = 1e300;
        *chunk = 1;
        for (int zc = std::min(g.n[2], 16); zc >= 1; --zc) {
            const long long items = tiles * ((g.n[2] + zc - 1) / zc);
            const double cost = (double)((items + slots - 1) / slots) * (zc + 1.0);
            if (cost < best) {
                best = cost;
                *chunk = zc;
            }
        }
        return best;
    };
    int v = U->variant, zc = U->zchunk;
    // the chosen variant, if it exists for this dtype, dimension and scheme
    const bool chosen = v >= 0 && sweep_smem(U->dtype, U->ndim, layout, scheme, v) > 0;
    if (!chosen) {
        // default: the packed pair kernel (FP32), else the first that fits
        v = sweep_smem(U->dtype, U->ndim, layout, scheme, kPairVariant) > 0 ? kPairVariant : -1;
        for (int c = 0; c < kNumSweepVariants && v < 0; ++c)
            if (sweep_smem(U->dtype, U->ndim, layout, scheme, c) > 0) v = c;
        if (v < 0) return fail(RIPPLE_ERR_INTERNAL, "no sweep kernel fits this configuration");
        // FP32 3D MUSCL-Hancock SoA fields: the row kernel where its wide tiles fill
        // the rounds (a plane of its 64 x 14 tile takes 3.8 us with one CTA per
        // SM, one of the pair kernel's 32 x 8 tile 2.3 us with two): 256^3 500
        // against 545 us a step, 150 x 101 x 131 106 against 95 us.  (AoS planes
        // staged in shared memory put a row's cells 20 bytes apart, so the row
        // kernel's loads of them conflict: 633 against 601 us at 256^3.)
        if (layout == LAYOUT_SOA && sweep_smem(U->dtype, U->ndim, layout, scheme, kRowVariant) > 0) {
            int zr, zp;
            if (3.8 * z_split(kRowVariant, &zr) < 2.3 * z_split(kPairVariant, &zp)) v = kRowVariant;
        }
        // a 2D grid with fewer tiles than SMs: the shorter tile spreads it over more SMs
        // (the one-cell-per-item 32x4 variant; FP64 arithmetic is the bound there)
        auto tiles = [&](int c) {
            return ((g.n[0] + kSweepVariants[c].tx - 1) / kSweepVariants[c].tx) *
                   ((g.n[1] + kSweepVariants[c].ty - 1) / kSweepVariants[c].ty);
        };
        if (U->ndim == 2 && U->dtype == RIPPLE_F64 && tiles(v) < ctx->sm_count &&
            sweep_smem(U->dtype, U->ndim, layout, scheme, 1) > 0 && tiles(1) > tiles(v))
            v = 1;
    }
    if (U->ndim == 3 && zc <= 0) z_split(v, &zc);
    const int tx = kSweepVariants[v].tx, ty = kSweepVariants[v].ty;
    const double inv_dx[3] = {1.0 / p->dx[0], 1.0 / p->dx[1], U->ndim == 3 ? 1.0 / p->dx[2] : 0.0};

    cudaStream_t s = ctx->stream;
    const bool params_changed = !U->prepared || U->prep_gamma != p->gamma || U->prep_bc != (int)p->bc ||
                                U->prep_dx[0] != p->dx[0] || U->prep_dx[1] != p->dx[1] ||
                                (U->ndim == 3 && U->prep_dx[2] != p->dx[2]);
    if (params_changed) {
        RIPPLE_CUDA(launch_prep(U->dtype, U->ndim, U->buf[U->cur], U->ctl, g, (int)p->bc, p->gamma, inv_dx,
                                (int)(U->steps_total % 3), 8 * ctx->sm_count, s));
        U->prepared = true;
        U->prep_gamma = p->gamma;
        U->prep_bc = (int)p->bc;
        for (int d = 0; d < 3; ++d) U->prep_dx[d] = p->dx[d];
    }

    SweepLaunch L{};
    L.sg.f = g;
    L.sg.tiles_x = (g.n[0] + tx - 1) / tx;
    L.sg.tiles_y = (g.n[1] + ty - 1) / ty;
    if (U->ndim == 3) {
        zc = std::min(zc, g.n[2]);
        L.sg.zchunk = zc;
        L.sg.chunks_z = (g.n[2] + zc - 1) / zc;
    } else {
        L.sg.zchunk = 1;
        L.sg.chunks_z = 1;
    }
    L.sg.items = L.sg.tiles_x * L.sg.tiles_y * L.sg.chunks_z;
    const int occ = std::max(1, sweep_occ(U->dtype, U->ndim, layout, scheme, v));
    L.grid = std::min(L.sg.items, occ * ctx->sm_count);
    L.ctl = U->ctl;
    L.stream = s;
    L.prm.gamma = p->gamma;
    L.prm.cfl = p->cfl;
    for (int d = 0; d < 3; ++d) L.prm.inv_dx[d] = inv_dx[d];
    L.prm.gamma_f = (float)p->gamma;
    L.prm.gm1_f = (float)(p->gamma - 1.0);
    for (int d = 0; d < 3; ++d) L.prm.inv_dx_f[d] = (float)inv_dx[d];
    L.prm.bc = (int)p->bc;

    // one launch per step (unsplit), or one sweep per axis (split: x, then y, then z;
    // each sweep writes the ghost images its successor reads; all read the same dt)
    const int sweeps = split ? U->ndim : 1;
    int64_t nsteps_left = nsteps;
    // several steps per launch unless a kernel was chosen: FP32 2D schemes and
    // the split step on strip walks; FP64 first-order 2D on compute-spread tiles
    // (per step, tiles of euler_sweep.cuh -> now: 64^2 17.5 -> 7.4 us, 256^2
    // 36 -> 19.7 us, 1024^2 380 -> 240 us)
    const bool walks = U->dtype == RIPPLE_F32 ? U->ndim == 2 || split : U->ndim == 2 && scheme == SCHEME_RUSANOV1;
    if (walks && !chosen) {
        st = walk_field_steps(U, *p, scheme, layout, nsteps);
        if (st != RIPPLE_OK) return st;
        nsteps_left = 0;
    }
    for (int64_t n = 0; n < nsteps_left; ++n) {
        for (int a = 0; a < sweeps; ++a) {
            const int in = U->cur, outb = 1 - U->cur;
            // the row kernel stages AoS planes through the grouped view and
            // stores its results directly (no output map)
            const bool rowk = v == kRowVariant;
            L.map_in = field_map(U, in, rowk && layout == LAYOUT_AOS ? 2 : 0, R, tx, ty, &st);
            if (!L.map_in) return st;
            L.map_out = rowk ? L.map_in : field_map(U, outb, 1, R, tx, ty, &st);
            if (!L.map_out) return st;
            L.out = U->buf[outb];
            L.prm.slot_in = (int)(U->steps_total % 3);
            L.prm.first = n == 0;
            L.prm.axis = split ? a : -1;
            L.prm.last = a == sweeps - 1;
            RIPPLE_CUDA(sweep_launch(U->dtype, U->ndim, layout, scheme, v, L));
            U->cur = outb;
        }
        U->steps_total++;
    }

    if (!stats) return RIPPLE_OK;
    // FP64 compensated totals of the final state
    const int nblocks = 2 * ctx->sm_count;
    const size_t pbytes = (size_t)nblocks * U->ncomp * 2 * sizeof(double);
    if (ctx->partials_bytes < pbytes) {
        RIPPLE_CUDA(cudaStreamSynchronize(s));
        ctx_free(ctx, ctx->partials, ctx->partials_bytes);
        ctx->partials = nullptr;
        ctx->partials_bytes = 0;
        st = ctx_alloc(ctx, pbytes, reinterpret_cast<void**>(&ctx->partials));
        if (st != RIPPLE_OK) return st;
        ctx->partials_bytes = round_up(pbytes, 256);
    }
    RIPPLE_CUDA(launch_totals(U->dtype, U->ncomp, U->buf[U->cur], g, ctx->partials, nblocks, U->ctl, s));
    RIPPLE_CUDA(cudaMemcpyAsync(ctx->h_ctl, U->ctl, sizeof(FieldCtl), cudaMemcpyDeviceToHost, s));
    RIPPLE_CUDA(cudaStreamSynchronize(s));
    const FieldCtl host = *ctx->h_ctl;
    stats->t = nsteps > 0 ? host.t : 0.0;
    stats->dt_last = nsteps > 0 ? host.dt_last : 0.0;
    for (int m = 0; m < 5; ++m) stats->totals[m] = m < U->ncomp ? host.totals[m] : 0.0;
    stats->steps_done = nsteps;
    if (host.err) {
        RIPPLE_CUDA(cudaMemsetAsync(&U->ctl->err, 0, sizeof(unsigned), s));
        RIPPLE_CUDA(cudaMemsetAsync(&U->ctl->counters[4], 0, 4 * sizeof(long long), s));
        return map_dev_err(host.err, &host);
    }
    return RIPPLE_OK;
}

}  // extern "C"
