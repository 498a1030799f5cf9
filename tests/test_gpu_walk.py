"""FP32 strip walks (2D Rusanov, MUSCL-Hancock and split FORCE steps, 3D split
FORCE steps; several steps per launch) against the FP64 oracle at the sizes
where a walk's edges fall: strips of 60 columns (64 in a z walk) with one, two
or an odd number of columns left, fields narrower than a pair or a halo,
single rows and planes, and more walks than resident warps."""
import numpy as np
import pytest

import inputs
import oracle
import paper_2104_08571_gb300 as R
from tests.gpu_util import LINF_F32, assert_parity, gpu_euler

pytestmark = pytest.mark.gpu
SCHEMES = {"rusanov": (R.RIPPLE_RUSANOV1, oracle.RUSANOV1), "mh": (R.RIPPLE_MUSCL_HANCOCK_MINMOD, oracle.MUSCL_HANCOCK),
           "force": (R.RIPPLE_FORCE_SPLIT, oracle.FORCE_SPLIT)}
BCS = [R.RIPPLE_BC_PERIODIC, R.RIPPLE_BC_TRANSMISSIVE]


@pytest.fixture(scope="module")
def ctx():
    import torch
    assert torch.cuda.is_available()
    c = R.ripple_ctx_create(0)
    R.use_torch_allocator(c, 0)
    yield c
    R.ripple_ctx_destroy(c)


def _state(dims, seed, amp=0.3):
    n, nd = int(np.prod(dims)), len(dims)
    r = inputs.uniform(seed, (nd + 2) * n).reshape((nd + 2,) + tuple(reversed(dims)))
    U = inputs.conserved(1.0 + amp * r[0], [amp * (r[1 + d] - 0.5) for d in range(nd)], 1.0 + amp * r[nd + 1])
    return U.astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("dims", [(2, 2), (3, 5), (59, 2), (60, 7), (61, 33), (62, 4), (63, 9), (64, 3), (120, 17),
                                  (121, 6), (5, 200)])
@pytest.mark.parametrize("scheme", sorted(SCHEMES))
@pytest.mark.parametrize("bc", BCS)
@pytest.mark.parametrize("layout", [R.RIPPLE_SOA, R.RIPPLE_AOS])
def test_walk_edges_2d(ctx, dims, scheme, bc, layout):
    U0 = _state(dims, seed=dims[0] * 7 + dims[1])
    got, st = gpu_euler(ctx, U0, 6, dtype=R.RIPPLE_F32, layout=layout, scheme=SCHEMES[scheme][0], bc=bc)
    ref, info = oracle.euler_run(U0, 6, scheme=SCHEMES[scheme][1], bc=bc)
    assert_parity(got, ref, 2e-5, LINF_F32)
    assert st["t"] == pytest.approx(info["t"], rel=1e-5)


@pytest.mark.parametrize("dims", [(1, 2, 3), (63, 2, 5), (64, 9, 8), (65, 3, 9), (60, 24, 17), (122, 25, 4)])
@pytest.mark.parametrize("bc", BCS)
@pytest.mark.parametrize("layout", [R.RIPPLE_SOA, R.RIPPLE_AOS])
def test_walk_edges_3d(ctx, dims, bc, layout):
    U0 = _state(dims, seed=dims[0] + 100 * dims[2])
    got, _ = gpu_euler(ctx, U0, 5, dtype=R.RIPPLE_F32, layout=layout, scheme=R.RIPPLE_FORCE_SPLIT, bc=bc)
    ref, _ = oracle.euler_run(U0, 5, scheme=oracle.FORCE_SPLIT, bc=bc)
    assert_parity(got, ref, 2e-5, LINF_F32)


def test_walks_handed_out_3d(ctx):
    """2,600 planes: more in-plane walks and more z walks than the GPU holds
    warps, so the later ones are handed out by the phase counters."""
    dims = (10, 13, 2600)
    U0 = _state(dims, seed=3)
    got, _ = gpu_euler(ctx, U0, 3, dtype=R.RIPPLE_F32, scheme=R.RIPPLE_FORCE_SPLIT, bc=R.RIPPLE_BC_PERIODIC)
    ref, _ = oracle.euler_run(U0, 3, scheme=oracle.FORCE_SPLIT, bc=oracle.PERIODIC)
    assert_parity(got, ref, 2e-5, LINF_F32)


@pytest.mark.parametrize("scheme", sorted(SCHEMES))
def test_walks_handed_out_2d(ctx, scheme):
    """2,500 x 7,900: more walks of at most 128 rows than warps; against the tiled pair kernel."""
    U0 = np.tile(_state((250, 790), seed=4), (1, 10, 10))
    a, _ = gpu_euler(ctx, U0, 2, dtype=R.RIPPLE_F32, scheme=SCHEMES[scheme][0], bc=R.RIPPLE_BC_PERIODIC)
    b, _ = gpu_euler(ctx, U0, 2, dtype=R.RIPPLE_F32, scheme=SCHEMES[scheme][0], bc=R.RIPPLE_BC_PERIODIC, variant=2)
    assert_parity(a, b.astype(np.float64), 1e-6, 1e-5)


@pytest.mark.parametrize("scheme", sorted(SCHEMES))
def test_walk_launches_of_a_long_call(ctx, scheme):
    """A call of more steps than one launch takes (256) equals two shorter calls on the same field, bit for bit."""
    U0 = inputs.euler2d_sine(70, ny=41).astype(np.float32)
    prm = R.make_fv_params([1.0 / 70, 1.0 / 41], scheme=SCHEMES[scheme][0])
    out = []
    for calls in ([300], [111, 189]):
        f = R.ripple_field_create(ctx, (70, 41), 4, R.RIPPLE_SOA, 2, R.RIPPLE_F32)
        R.ripple_field_upload(f, U0)
        for n in calls:
            assert R.ripple_fv_step(f, prm, n)["steps_done"] == n
        out.append(R.ripple_field_download(f))
        R.ripple_field_destroy(f)
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("where", [(0, 0), (61, 3), (69, 40)])
@pytest.mark.parametrize("scheme", sorted(SCHEMES))
def test_walk_reports_a_bad_cell(ctx, scheme, where):
    U0 = inputs.uniform_state((70, 41), 1.0, [0.1, 0.0], 1.0)
    U0[3, where[1], where[0]] = -1.0
    with pytest.raises(R.RippleError) as ei:
        gpu_euler(ctx, U0, 1, dtype=R.RIPPLE_F32, scheme=SCHEMES[scheme][0], bc=R.RIPPLE_BC_TRANSMISSIVE)
    assert ei.value.status == R.RIPPLE_ERR_NUMERIC
