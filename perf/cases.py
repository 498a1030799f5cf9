"""Performance cases of the stencil library: what its users run, through its public entry points.

A case is a dict of plain values.  Four kinds cover the paths of the library:

  kind "fv"      a whole Euler solve on one field: the state goes into the
                 field from device memory, ``ripple_fv_step`` advances it, the
                 state comes back to device memory (and, with "stats", the
                 simulated time and the conserved totals to the host).
  kind "eik"     a whole eikonal solve on one field: slowness in, travel times out.
  kind "batch"   many uneven 2D Euler problems on page-locked host arrays,
                 submitted at once to the batch runtime.
  kind "mix"     a burst of Euler and eikonal requests on pageable host arrays,
                 served by the batch runtime's continuous batching.

Every input is made from the seed alone: the library's workload states (sine
density wave, spherical blast with noise, log-normal slowness), with seeded
amplitudes, phases, noise and sources.
"""
import math
import random

import numpy as np
import torch

import paper_2104_08571_gb300 as R

GAMMA, CFL = 1.4, 0.4

SCHEMES = {"rusanov": R.RIPPLE_RUSANOV1, "mh": R.RIPPLE_MUSCL_HANCOCK_MINMOD, "force": R.RIPPLE_FORCE_SPLIT}
LAYOUTS = {"soa": R.RIPPLE_SOA, "aos": R.RIPPLE_AOS}
BCS = {"periodic": R.RIPPLE_BC_PERIODIC, "transmissive": R.RIPPLE_BC_TRANSMISSIVE}
DTYPES = {"f32": (R.RIPPLE_F32, torch.float32), "f64": (R.RIPPLE_F64, torch.float64)}


def _fv(name, nx, ny, nz, scheme, bc, layout, dtype, steps, stats):
    c = {"kind": "fv", "nx": nx, "ny": ny, "nz": nz, "scheme": scheme, "bc": bc, "layout": layout, "dtype": dtype,
         "steps": steps, "stats": stats}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the headline workload: a 3D blast at 256^3, second order, single precision
        _fv("mh3d_256", 256, 256, 256, "mh", "transmissive", "soa", "f32", 20, False),
        # a production domain that fits no tile, in the record layout, periodic
        _fv("mh3d_aos_odd", 150, 101, 131, "mh", "periodic", "aos", "f32", 20, False),
        # a coarse 3D run (parameter scans, coarse levels): few tiles, many steps
        _fv("mh3d_48", 48, 48, 48, "mh", "transmissive", "soa", "f32", 40, True),
        # a 2D second-order run on a rectangular domain
        _fv("mh2d_odd", 1000, 701, 0, "mh", "transmissive", "soa", "f32", 30, False),
        # the double-precision reference workload: 128^2, first order, 100 steps, with its totals
        _fv("rus2d_f64_128", 128, 128, 0, "rusanov", "periodic", "soa", "f64", 100, True),
        # the smallest calls: a coarse problem advanced a few steps at a time, its time read back every call
        _fv("rus2d_64_short", 64, 64, 0, "rusanov", "periodic", "soa", "f32", 4, True),
        # the paper's own solver (split FORCE) on a large 2D grid
        _fv("force2d_4096", 4096, 4096, 0, "force", "periodic", "soa", "f32", 10, False),
        # the paper's own solver in 3D, ragged on every axis
        _fv("force3d_odd", 200, 171, 186, "force", "transmissive", "soa", "f32", 10, False),
        # travel times on the 2D and 3D workload grids
        {"name": "eik2d_2048", "kind": "eik", "nx": 2048, "ny": 2048, "nz": 0, "dtype": "f32", "nsrc": 2},
        {"name": "eik3d_192", "kind": "eik", "nx": 192, "ny": 192, "nz": 192, "dtype": "f32", "nsrc": 2},
        # the batched workload: 512 uneven problems of 100 steps
        {"name": "batch_512", "kind": "batch", "count": 512, "lo": 32, "hi": 512, "steps": 100, "sizes": 1},
        # a burst of served requests, 70 % Euler and 30 % eikonal
        {"name": "mix_24", "kind": "mix", "count": 24, "lo": 64, "hi": 1024, "steps": 500, "sizes": 1},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fv3", "fv3", "fv2", "fv2", "fv2", "eik", "eik", "batch", "mix"])
    if kind in ("fv3", "fv2"):
        dtype = "f64" if rng.random() < 0.25 else "f32"
        # the split solver runs in single precision in 3D, in both in 2D
        scheme = rng.choice(["mh", "mh", "rusanov", "rusanov" if kind == "fv3" and dtype == "f64" else "force"])
        bc, layout = rng.choice(sorted(BCS)), rng.choice(["soa", "soa", "aos"])
        if kind == "fv3":
            nx, ny, nz = (_log(rng, 20, 256) for _ in range(3))
            cap = 2e8
        else:
            nx, ny, nz = _log(rng, 32, 4096), _log(rng, 32, 4096), 0
            cap = 1.6e8
        most = cap / (nx * ny * max(1, nz)) / (8 if dtype == "f64" else 1)
        steps = max(1, min(_log(rng, 4, 100), int(most)))
        return _fv(None, nx, ny, nz, scheme, bc, layout, dtype, steps, rng.random() < 0.4)
    if kind == "eik":
        dtype = "f64" if rng.random() < 0.2 else "f32"
        most = 1400 if dtype == "f64" else 2048
        if rng.random() < 0.5:
            dims = (_log(rng, 64, most), _log(rng, 64, most), 0)
        else:
            dims = tuple(_log(rng, 24, 150 if dtype == "f64" else 192) for _ in range(3))
        return {"kind": "eik", "nx": dims[0], "ny": dims[1], "nz": dims[2], "dtype": dtype, "nsrc": rng.randint(1, 4)}
    if kind == "batch":
        return {"kind": "batch", "count": _log(rng, 16, 512), "lo": 32, "hi": _log(rng, 64, 512),
                "steps": _log(rng, 20, 100), "sizes": rng.randrange(1 << 20)}
    return {"kind": "mix", "count": rng.randint(4, 24), "lo": 64, "hi": _log(rng, 200, 900),
            "steps": _log(rng, 60, 500), "sizes": rng.randrange(1 << 20)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gen(seed, salt=0):
    g = torch.Generator(device=_device())
    g.manual_seed((seed * 1000003 + salt * 7919 + 17) % (1 << 62))
    return g


def _dims(case):
    return tuple(case[k] for k in ("nx", "ny", "nz") if case[k])


def _axes(dims):
    """Cell centres of every axis on (0, 1), shaped to broadcast over (z, y, x)."""
    nd = len(dims)
    out = []
    for d, n in enumerate(dims):
        shape = [1] * nd
        shape[nd - 1 - d] = n
        out.append(((torch.arange(n, device=_device(), dtype=torch.float64) + 0.5) / n).reshape(shape))
    return out


def _conserved(rho, vel, p):
    ke = sum(0.5 * rho * u * u for u in vel)
    E = p / (GAMMA - 1.0) + ke
    return torch.stack([rho] + [rho * u for u in vel] + [E.expand_as(rho)])


def _sine(dims, seed, salt=0):
    """An advected density wave, seeded amplitude, phases and velocity, 1 % noise on the density."""
    r = random.Random(seed * 7919 + salt)
    amp, ph = r.uniform(0.05, 0.3), [r.random() for _ in dims]
    ax = _axes(dims)
    w = 1.0
    for a, p in zip(ax, ph):
        w = w * torch.sin(2.0 * math.pi * (a + p))
    noise = torch.rand(tuple(reversed(dims)), generator=_gen(seed, salt), device=_device(), dtype=torch.float64)
    rho = (1.0 + amp * w) * (1.0 + 0.01 * (2.0 * noise - 1.0))
    vel = [torch.full_like(rho, v * r.uniform(0.8, 1.2)) for v in (1.0, 0.5, 0.25)[: len(dims)]]
    return _conserved(rho, vel, torch.ones_like(rho))


def _blast(dims, seed, salt=0):
    """A spherical blast around the centre, 1 % noise on the density."""
    r2 = sum((a - 0.5) ** 2 for a in _axes(dims))
    inside = r2 < 0.04
    noise = torch.rand(tuple(reversed(dims)), generator=_gen(seed, salt), device=_device(), dtype=torch.float64)
    rho = torch.where(inside, 1.0, 0.125).to(torch.float64) * (1.0 + 0.01 * (2.0 * noise - 1.0))
    p = torch.where(inside, 1.0, 0.1).to(torch.float64)
    return _conserved(rho, [torch.zeros_like(rho) for _ in dims], p)


def _slowness(dims, seed, salt=0):
    """exp(0.5 g), g Gaussian noise under a periodic 3-wide box mean."""
    g = torch.randn(tuple(reversed(dims)), generator=_gen(seed, salt), device=_device(), dtype=torch.float64)
    for d in range(g.ndim):
        g = (g + torch.roll(g, 1, d) + torch.roll(g, -1, d)) / 3.0
    return torch.exp(0.5 * g)


def _sources(dims, count, seed, salt=0):
    r = random.Random(seed * 104729 + salt)
    got = []
    while len(got) < count:
        c = tuple(r.randrange(n) for n in dims)
        if c not in got:
            got.append(c)
    return got


def _fv_input(case, seed):
    """The initial state as the library gets it: the field's type, component-major."""
    U = (_sine if case["bc"] == "periodic" else _blast)(_dims(case), seed)
    return U.to(DTYPES[case["dtype"]][1])


def _requests(case):
    """The sizes of a batch's or a burst's requests: fixed by the case, not by the seed."""
    r = random.Random(case["sizes"])
    out = []
    for k in range(case["count"]):
        if case["kind"] == "batch" or r.random() < 0.7:
            side = min(case["hi"], max(case["lo"], int(math.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"]))))))
            steps = case["steps"] if case["kind"] == "batch" else r.randint(max(1, case["steps"] // 10), case["steps"])
            out.append({"euler": True, "side": side, "steps": steps})
        else:
            lo = min(128, case["hi"])
            side = min(case["hi"], int(math.exp(r.uniform(math.log(lo), math.log(case["hi"])))))
            out.append({"euler": False, "side": side, "nsrc": r.randint(1, 4)})
    return out


def _request_input(q, seed, k):
    dims = (q["side"], q["side"])
    return (_sine(dims, seed, k) if q["euler"] else _slowness(dims, seed, k)).to(torch.float32)


SLAB = 32  # problems of a batch that share one page-locked array


# ---------------------------------------------------------------------------
# the library's handles
# ---------------------------------------------------------------------------
_contexts = {}


def _context(kind):
    """One context per kind of work, as a program keeps it: fields on a PyTorch stream and allocator, or a batch runtime."""
    if kind not in _contexts:
        ctx = R.ripple_ctx_create(0, 0 if kind == "field" else 40 << 30)
        if kind == "field":
            R.use_torch_allocator(ctx, 0)
            stream = torch.cuda.Stream()
            R.ripple_set_stream(ctx, stream)
            _contexts[kind] = (ctx, stream)
        else:
            if kind == "batch":
                R.ripple_batch_configure(ctx, steps_per_sync=100, use_graphs=True, staging=2)
            else:
                R.ripple_batch_configure(ctx, steps_per_sync=8, use_graphs=True, active_cells=4 << 20)
            _contexts[kind] = (ctx, None)
    return _contexts[kind][0]


class _State:
    """A case's inputs, outputs and handles; the fields go with it."""

    def __init__(self, case):
        self.case = case
        self.fields = []

    def __del__(self):
        for f in self.fields:
            R.ripple_field_destroy(f)


def prepare(case, seed):
    s = _State(case)
    if case["kind"] == "fv":
        dims, nd = _dims(case), len(_dims(case))
        ctx = _context("field")
        U = _fv_input(case, seed)
        if case["layout"] == "aos":
            U = torch.movedim(U, 0, -1)
        s.U = U.contiguous()
        s.out = torch.empty_like(s.U)
        torch.cuda.synchronize()  # the library works on its own stream: what made the inputs is done
        s.layout = LAYOUTS[case["layout"]]
        s.field = R.ripple_field_create(ctx, dims, nd + 2, s.layout, 2 if case["scheme"] == "mh" else 1,
                                        DTYPES[case["dtype"]][0])
        s.fields.append(s.field)
        s.params = R.make_fv_params([1.0 / n for n in dims], GAMMA, CFL, SCHEMES[case["scheme"]], BCS[case["bc"]])
    elif case["kind"] == "eik":
        dims = _dims(case)
        ctx = _context("field")
        dt, tt = DTYPES[case["dtype"]]
        s.slow = _slowness(dims, seed).to(tt).contiguous()
        s.out = torch.empty_like(s.slow)
        torch.cuda.synchronize()
        s.sources = _sources(dims, case["nsrc"], seed)
        s.h = 1.0 / max(dims)
        s.fs = R.ripple_field_create(ctx, dims, 1, R.RIPPLE_SOA, 0, dt)
        s.fields.append(s.fs)
        s.ft = R.ripple_field_create(ctx, dims, 1, R.RIPPLE_SOA, 1, dt)
        s.fields.append(s.ft)
    else:
        s.ctx = _context(case["kind"])
        s.requests, s.outputs = [], []
        qs = _requests(case)
        pinned = case["kind"] == "batch"
        for at in range(0, len(qs), SLAB if pinned else 1):
            part = qs[at: at + (SLAB if pinned else 1)]
            ins = [_request_input(q, seed, at + i) for i, q in enumerate(part)]
            flat = torch.cat([x.reshape(-1) for x in ins])
            host_in = torch.empty(flat.numel(), dtype=torch.float32, pin_memory=pinned)
            host_in.copy_(flat)
            host_out = torch.zeros(flat.numel(), dtype=torch.float32, pin_memory=pinned)
            s.outputs.append(host_out)
            a = 0
            for i, (q, x) in enumerate(zip(part, ins)):
                n, shape = x.numel(), tuple(x.shape)
                src, dst = host_in[a: a + n].numpy().reshape(shape), host_out[a: a + n].numpy().reshape(shape)
                a += n
                if q["euler"]:
                    s.requests.append(R.euler_request(src, q["steps"], [1.0 / q["side"]] * 2, GAMMA, CFL,
                                                      R.RIPPLE_BC_PERIODIC, out=dst))
                else:
                    where = _sources((q["side"],) * 2, q["nsrc"], seed, at + i)
                    s.requests.append(R.eikonal_request(src, where, 1.0 / q["side"], 1e-6, out=dst))
    torch.cuda.synchronize()
    return s


def run(s):
    case = s.case
    if case["kind"] == "fv":
        R.ripple_field_upload(s.field, s.U, s.layout)
        st = R.ripple_fv_step(s.field, s.params, case["steps"], stats=case["stats"])
        R.ripple_field_download(s.field, s.layout, out=s.out)
        if st is None:
            return {"state": s.out}
        real = np.float32 if case["dtype"] == "f32" else np.float64
        return {"state": s.out, "time": np.array([st["t"], st["dt_last"]], dtype=real),
                "totals": np.array(st["totals"][: len(_dims(case)) + 2], dtype=real)}
    if case["kind"] == "eik":
        R.ripple_field_upload(s.fs, s.slow)
        R.ripple_eikonal_solve(s.fs, s.ft, s.sources, s.h, 1e-6)
        R.ripple_field_download(s.ft, R.RIPPLE_SOA, out=s.out.unsqueeze(0))
        return {"T": s.out}
    for t in R.ripple_batch_submit(s.ctx, s.requests):
        info = R.ripple_wait(s.ctx, t)
        if info["status"] != R.RIPPLE_OK:
            raise RuntimeError("request failed with status %d" % info["status"])
    return s.outputs


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
# floating-point operations of one cell update: per axis one face (physical
# fluxes of both states, wave speeds, dissipation), the update, the CFL term;
# second order adds the slopes and the predicted states, FORCE the Richtmyer
# state and its flux
FLOPS = {"rusanov": {2: 110, 3: 190}, "mh": {2: 330, 3: 620}, "force": {2: 150, 3: 280}}


def work(case):
    """One read and one write of the state per step (each step's input is the whole result of the step before:
    its dt is a maximum over all of it), and the copies in and out; an eikonal cell is updated at least once."""
    if case["kind"] == "fv":
        dims = _dims(case)
        nd, cells, es = len(dims), math.prod(dims), 4 if case["dtype"] == "f32" else 8
        return {"bytes": 2.0 * cells * (nd + 2) * es * (case["steps"] + 2),
                "flops": float(cells * case["steps"] * FLOPS[case["scheme"]][nd])}
    if case["kind"] == "eik":
        dims = _dims(case)
        cells, es = math.prod(dims), 4 if case["dtype"] == "f32" else 8
        return {"bytes": 2.0 * cells * es * 3, "flops": float(cells * (12 if len(dims) == 2 else 30))}
    b = f = 0.0
    for q in _requests(case):
        cells = q["side"] ** 2
        if q["euler"]:
            b += 2.0 * cells * 16 * (q["steps"] + 2)
            f += cells * q["steps"] * FLOPS["rusanov"][2]
        else:
            b += 2.0 * cells * 4 * 3
            f += cells * 12.0
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# the same results in 64 bits, by plain tensor operations
# ---------------------------------------------------------------------------
def _prim(U, nd):
    rho = U[0]
    u = [U[1 + d] / rho for d in range(nd)]
    p = (GAMMA - 1.0) * (U[nd + 1] - 0.5 * sum(U[1 + d] * u[d] for d in range(nd)))
    return rho, u, p


def _flux(U, d, nd):
    """Physical flux along axis d, and |u_d| + c."""
    rho, u, p = _prim(U, nd)
    F = U * u[d]
    F[1 + d] += p
    F[nd + 1] += p * u[d]
    return F, u[d].abs() + torch.sqrt(GAMMA * p / rho)


def _speed(U, dx, nd):
    rho, u, p = _prim(U, nd)
    c = torch.sqrt(GAMMA * p / rho)
    return float(sum((u[d].abs() + c) / dx[d] for d in range(nd)).max())


def _pad(U, axis, n, bc):
    """n ghost layers on both ends of one axis."""
    size = U.shape[axis]
    if bc == "periodic":
        return torch.cat([U.narrow(axis, size - n, n), U, U.narrow(axis, 0, n)], axis)
    lo, hi = U.narrow(axis, 0, 1), U.narrow(axis, size - 1, 1)
    return torch.cat([lo] * n + [U] + [hi] * n, axis)


def _rusanov(L, Rt, d, nd):
    FL, sL = _flux(L, d, nd)
    FR, sR = _flux(Rt, d, nd)
    return 0.5 * (FL + FR) - 0.5 * torch.maximum(sL, sR) * (Rt - L)


def _force(L, Rt, d, nd, r):
    FL, _ = _flux(L, d, nd)
    FR, _ = _flux(Rt, d, nd)
    RI, _ = _flux(0.5 * (L + Rt) - 0.5 * r * (FR - FL), d, nd)
    return 0.25 * (FL + 2.0 * RI + FR - (Rt - L) / r)


def _advance(U, dx, scheme, bc, steps):
    """`steps` steps of a component-major state (ncomp, [z,] y, x); returns it, the time and the last dt."""
    nd = U.ndim - 1
    t = dt = 0.0
    for _ in range(steps):
        dt = CFL / _speed(U, dx, nd)
        t += dt
        new = U if scheme == "force" else U.clone()
        for d in range(nd):
            axis, n, r = U.ndim - 1 - d, U.shape[U.ndim - 1 - d], dt / dx[d]
            if scheme == "mh":
                P = _pad(U, axis, 2, bc)
                D = P.narrow(axis, 1, n + 3) - P.narrow(axis, 0, n + 3)
                a, b = D.narrow(axis, 0, n + 2), D.narrow(axis, 1, n + 2)
                half = 0.25 * (torch.sign(a) + torch.sign(b)) * torch.minimum(a.abs(), b.abs())
                del D, a, b
                C = P.narrow(axis, 1, n + 2)
                lo, hi = C - half, C + half
                del half
                move = 0.5 * r * (_flux(lo, d, nd)[0] - _flux(hi, d, nd)[0])
                lo += move
                hi += move
                del move, P, C
                F = _rusanov(hi.narrow(axis, 0, n + 1), lo.narrow(axis, 1, n + 1), d, nd)
                del lo, hi
            else:
                P = _pad(new if scheme == "force" else U, axis, 1, bc)
                L, Rt = P.narrow(axis, 0, n + 1), P.narrow(axis, 1, n + 1)
                F = _force(L, Rt, d, nd, r) if scheme == "force" else _rusanov(L, Rt, d, nd)
            new = new - r * (F.narrow(axis, 1, n) - F.narrow(axis, 0, n))
        U = new
    return U, t, dt


def _travel_times(slow, sources, h):
    """The fixed point of the upwind update under simultaneous sweeps."""
    nd = slow.ndim
    inf = math.inf
    f = slow * h
    P = torch.full([n + 2 for n in slow.shape], inf, dtype=torch.float64, device=slow.device)
    T = P
    for d in range(nd):
        T = T.narrow(d, 1, slow.shape[d])
    at = tuple(torch.tensor([c[nd - 1 - d] for c in sources], device=slow.device) for d in range(nd))
    T[at] = 0.0

    def near(d):
        Q = P
        for e in range(nd):
            if e != d:
                Q = Q.narrow(e, 1, slow.shape[e])
        n = slow.shape[d]
        return torch.minimum(Q.narrow(d, 0, n), Q.narrow(d, 2, n))

    big = 1e30
    for k in range(1, 40001):
        if nd == 2:
            a, b = near(0), near(1)
            lo, hi = torch.minimum(a, b).clamp_max(big), torch.maximum(a, b).clamp_max(big)
            gap = hi - lo
            g = torch.where(gap >= f, lo + f, 0.5 * (lo + hi + torch.sqrt((2.0 * f * f - gap * gap).clamp_min(0.0))))
        else:
            u, v, w = near(0).clamp_max(big), near(1).clamp_max(big), near(2).clamp_max(big)
            a, c = torch.minimum(u, v), torch.maximum(u, v)
            b = torch.maximum(a, torch.minimum(c, w))
            a, c = torch.minimum(a, w), torch.maximum(c, w)
            g = a + f
            two = 0.5 * (a + b + torch.sqrt((2.0 * f * f - (b - a) ** 2).clamp_min(0.0)))
            s = a + b + c
            three = (s + torch.sqrt((3.0 * f * f - ((b - a) ** 2 + (c - a) ** 2 + (c - b) ** 2)).clamp_min(0.0))) / 3.0
            g = torch.where(g > b, two, g)
            g = torch.where((a + f > b) & (two > c), three, g)
        new = torch.minimum(T, g)
        if k % 64 == 0 and bool(((T - new).abs() <= 1e-15 * new).logical_or(T == new).all()):
            break
        T.copy_(new)
    return T


def exact(case, seed):
    if case["kind"] == "fv":
        dims = _dims(case)
        U = _fv_input(case, seed).to(torch.float64)
        U, t, dt = _advance(U, [1.0 / n for n in dims], case["scheme"], case["bc"], case["steps"])
        totals = U.reshape(U.shape[0], -1).sum(1).cpu().numpy()
        state = (torch.movedim(U, 0, -1) if case["layout"] == "aos" else U).contiguous()
        return {"state": state, "time": np.array([t, dt]), "totals": totals} if case["stats"] else {"state": state}
    if case["kind"] == "eik":
        dims = _dims(case)
        slow = _slowness(dims, seed).to(DTYPES[case["dtype"]][1]).to(torch.float64)
        T = _travel_times(slow, _sources(dims, case["nsrc"], seed), 1.0 / max(dims))
        return {"T": T.contiguous()}
    # the first arrays of a batch; of a burst, every request
    out, left = [], 64
    qs = _requests(case)
    for at in range(0, len(qs), SLAB if case["kind"] == "batch" else 1):
        part = qs[at: at + (SLAB if case["kind"] == "batch" else 1)]
        if len(part) > left:
            out.append(None)
            continue
        left -= len(part)
        got = []
        for i, q in enumerate(part):
            x = _request_input(q, seed, at + i).to(torch.float64)
            if q["euler"]:
                x = _advance(x, [1.0 / q["side"]] * 2, "rusanov", "periodic", q["steps"])[0]
            else:
                x = _travel_times(x, _sources((q["side"],) * 2, q["nsrc"], seed, at + i), 1.0 / q["side"])
            got.append(x.reshape(-1))
        out.append(torch.cat(got).cpu())
    return out
