"""Non-admissible states that a multi-step kernel itself produces (every cell of
the input is admissible): the one cell that a step leaves with negative
pressure is named, wherever it lies on strips, segments and tiles; states that
are negative only between two sweeps of the split step, or only on a
reconstructed face, are reported although every updated cell is admissible;
and the same states at a Courant number of 0.4 are not reported at all.

A step of the oracle says the same: one non-admissible cell in its result, or
its NUMERIC status."""
import numpy as np
import pytest

import inputs
import oracle
import paper_2104_08571_gb300 as R

pytestmark = pytest.mark.gpu
SCHEMES = {"rusanov": (R.RIPPLE_RUSANOV1, oracle.RUSANOV1), "mh": (R.RIPPLE_MUSCL_HANCOCK_MINMOD, oracle.MUSCL_HANCOCK),
           "force": (R.RIPPLE_FORCE_SPLIT, oracle.FORCE_SPLIT)}
X2, Y2 = (0, 1, 7, 8, 31, 32, 58, 59, 60, 61, 118, 119, 120), (0, 1, 19, 20, 38, 39)
X3, Y3, Z3 = (0, 1, 59, 60, 63, 64, 127, 128, 129), (0, 5, 10), (0, 7, 8, 18)
# density, pressure and velocity of one cell in a gas of density and pressure 1 at rest, the Courant number of the
# step, and where the bad state lies from that cell
HOT = (1.0, 10.0, (0, 0), 2.0, (0, 0))
FORCE2 = (3.25, 0.2, (0.5, 1), 3.5, (1, 0))
FORCE2_BETWEEN = (0.84, 6.6, (0.5, 1), 4.1, (0, 0))
FORCE3 = (4.0, 0.22, (0, 0, 1), 5.9, (0, 0, 0))
FORCE3_AFTER_X = (1.23, 6.1, (-1, -1, -1), 5.4, (0, 0, 0))
FORCE3_AFTER_Y = (5.4, 0.23, (1, -1, -0.5), 3.77, (1, 0, 0))


@pytest.fixture(scope="module")
def ctx():
    c = R.ripple_ctx_create(0)
    yield c
    R.ripple_ctx_destroy(c)


def _places(dims):
    """Every x of the list with the other coordinates in turn."""
    if len(dims) == 2:
        return [(x, Y2[i % len(Y2)]) for i, x in enumerate(X2)]
    return [(x, Y3[i % len(Y3)], Z3[i % len(Z3)]) for i, x in enumerate(X3)]


def _one_cell(dims, at, cell):
    """The gas at rest with the special cell placed so that the bad state falls on `at` (periodic)."""
    rho, p, u, _, off = cell
    nd = len(dims)
    U = inputs.uniform_state(dims, 1.0, [0.0] * nd, 1.0)
    c = tuple(reversed([(at[d] - off[d]) % dims[d] for d in range(nd)]))
    for m, v in enumerate([rho] + [rho * x for x in u] + [p / 0.4 + 0.5 * rho * sum(x * x for x in u)]):
        U[(m,) + c] = v
    return U


def _bad_cells(U):
    nd = U.shape[0] - 2
    p = U[-1] - 0.5 * (U[1:1 + nd] ** 2).sum(0) / U[0]
    return [tuple(int(v) for v in reversed(c)) for c in np.argwhere(~((U[0] > 0) & (p > 0)))]


def _step(ctx, U, scheme, bc, dtype, layout, cfl, steps=1):
    dims = tuple(reversed(U.shape[1:]))
    f = R.ripple_field_create(ctx, dims, U.shape[0], layout, 2, dtype)
    try:
        R.ripple_field_upload(f, np.ascontiguousarray(U, dtype=np.float32 if dtype == R.RIPPLE_F32 else np.float64))
        R.ripple_fv_step(f, R.make_fv_params([1 / 48] * len(dims), cfl=cfl, scheme=scheme, bc=bc), steps)
    finally:
        R.ripple_field_destroy(f)


def _oracle(U, scheme, bc, cfl):
    return oracle.euler_run(U, 1, cfl=cfl, dx=[1 / 48] * (U.ndim - 1), scheme=scheme, bc=bc, allow_numeric=True)


CELL = [("rusanov", (121, 40), HOT, R.RIPPLE_F32), ("mh", (121, 40), HOT, R.RIPPLE_F32), ("force", (121, 40), FORCE2, R.RIPPLE_F32),
        ("force", (130, 11, 19), FORCE3, R.RIPPLE_F32), ("rusanov", (121, 40), HOT, R.RIPPLE_F64)]


@pytest.mark.parametrize("scheme,dims,cell,dtype", CELL)
@pytest.mark.parametrize("layout", [R.RIPPLE_SOA, R.RIPPLE_AOS])
def test_the_bad_cell_of_a_step_is_named(ctx, scheme, dims, cell, dtype, layout):
    for at in _places(dims):
        U = _one_cell(dims, at, cell)
        ref, info = _oracle(U, SCHEMES[scheme][1], oracle.PERIODIC, cell[3])
        assert not _bad_cells(U)
        # (the oracle's split step checks its result itself and then returns no new state)
        assert info["status"] == oracle.NUMERIC if scheme == "force" else _bad_cells(ref) == [at]
        with pytest.raises(R.RippleError) as ei:
            _step(ctx, U, SCHEMES[scheme][0], R.RIPPLE_BC_PERIODIC, dtype, layout, cell[3])
        assert ei.value.status == R.RIPPLE_ERR_NUMERIC
        where = ", ".join(str(v) for v in at + (0,) * (3 - len(at)))
        assert f"updated cell ({where})" in str(ei.value), (at, str(ei.value))
        for bc in (R.RIPPLE_BC_PERIODIC, R.RIPPLE_BC_TRANSMISSIVE):
            _step(ctx, U, SCHEMES[scheme][0], bc, dtype, layout, 0.4, 3)


@pytest.mark.parametrize("dims,cell", [((121, 40), FORCE2_BETWEEN), ((130, 11, 19), FORCE3_AFTER_X), ((130, 11, 19), FORCE3_AFTER_Y)])
@pytest.mark.parametrize("layout", [R.RIPPLE_SOA, R.RIPPLE_AOS])
def test_a_bad_state_between_two_sweeps_is_reported(ctx, dims, cell, layout):
    for at in _places(dims):
        U = _one_cell(dims, at, cell)
        assert not _bad_cells(U)
        assert _oracle(U, oracle.FORCE_SPLIT, oracle.PERIODIC, cell[3])[1]["status"] == oracle.NUMERIC
        with pytest.raises(R.RippleError) as ei:
            _step(ctx, U, R.RIPPLE_FORCE_SPLIT, R.RIPPLE_BC_PERIODIC, R.RIPPLE_F32, layout, cell[3])
        assert ei.value.status == R.RIPPLE_ERR_NUMERIC and "state in the tile" in str(ei.value), (at, str(ei.value))


@pytest.mark.parametrize("layout", [R.RIPPLE_SOA, R.RIPPLE_AOS])
@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("sign", [1, -1])
def test_a_bad_face_state_is_reported(ctx, layout, axis, sign):
    """Momenta 0, 2, 4 at a pressure of 0.01: the middle cell's extrapolated state has more kinetic than total
    energy (the momentum's slope is 2, the energy's too), and in a step of 1e-4 no cell changes much."""
    dims = (121, 40)
    n = dims[axis]
    for i in [v for v in (X2 if axis == 0 else Y2) if 1 <= v <= n - 2]:
        m = np.where(np.arange(n) < i, 0.0, np.where(np.arange(n) == i, 2.0, 4.0))
        if sign < 0:
            m = m[::-1]
        shape = [1, n] if axis == 0 else [n, 1]
        U = np.zeros((4,) + tuple(reversed(dims)))
        U[0] = 1.0
        U[1 + axis] = m.reshape(shape)
        U[3] = 0.01 / 0.4 + 0.5 * U[1 + axis] ** 2
        assert not _bad_cells(U)
        assert _oracle(U, oracle.MUSCL_HANCOCK, oracle.TRANSMISSIVE, 1e-4)[1]["status"] == oracle.NUMERIC
        with pytest.raises(R.RippleError) as ei:
            _step(ctx, U, R.RIPPLE_MUSCL_HANCOCK_MINMOD, R.RIPPLE_BC_TRANSMISSIVE, R.RIPPLE_F32, layout, 1e-4)
        assert ei.value.status == R.RIPPLE_ERR_NUMERIC and "state in the tile" in str(ei.value), (i, str(ei.value))


@pytest.mark.parametrize("dims,cfg", [((121, 40), {"staging": 0, "solo_rounds": False}), ((121, 40), {"staging": 1, "solo_rounds": False}),
                                      ((121, 40), {"staging": 2, "solo_rounds": False, "async_queue": True}),
                                      ((121, 40), {"solo_rounds": True}), ((420, 400), {"solo_rounds": True})])
def test_a_served_bad_step_is_reported(ctx, dims, cfg):
    R.ripple_batch_configure(ctx, **cfg)
    places = _places(dims) + [(x, y) for x in (dims[0] - 1, dims[0] - 2) for y in (0, dims[1] - 1)]
    for cfl, want in ((2.0, R.RIPPLE_ERR_NUMERIC), (0.4, R.RIPPLE_OK)):
        reqs = [R.euler_request(_one_cell(dims, at, HOT).astype(np.float32), 1, [1 / 48] * 2, cfl=cfl) for at in places]
        got = [R.ripple_wait(ctx, t, 60000)["status"] for t in R.ripple_batch_submit(ctx, reqs)]
        assert got == [want] * len(places)
