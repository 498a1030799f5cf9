"""FP64 first-order 2D steps (several per launch, tile sides chosen by the
field's size) against the oracle: one-cell grids, sides that cut a tile to one
row or column, and grids whose tiles outnumber the resident CTAs."""
import numpy as np
import pytest

import inputs
import oracle
import paper_2104_08571_gb300 as R
from tests.gpu_util import LINF_F64, assert_parity, gpu_euler

pytestmark = pytest.mark.gpu
BCS = [R.RIPPLE_BC_PERIODIC, R.RIPPLE_BC_TRANSMISSIVE]


@pytest.fixture(scope="module")
def ctx():
    c = R.ripple_ctx_create(0)
    yield c
    R.ripple_ctx_destroy(c)


def _state(dims, amp=0.3):
    n = int(np.prod(dims))
    r = inputs.uniform(dims[0] * 7 + dims[1], 4 * n).reshape((4,) + tuple(reversed(dims)))
    return inputs.conserved(1.0 + amp * r[0], [amp * (r[1] - 0.5), amp * (r[2] - 0.5)], 1.0 + amp * r[3])


@pytest.mark.parametrize("dims", [(1, 1), (1, 7), (2, 3), (8, 4), (9, 5), (16, 33), (128, 7), (129, 113), (333, 2),
                                  (5, 700), (701, 333)])
@pytest.mark.parametrize("bc", BCS)
def test_tile_edges(ctx, dims, bc):
    U0 = _state(dims)
    ref, info = oracle.euler_run(U0, 6, scheme=oracle.RUSANOV1, bc=bc)
    got = [gpu_euler(ctx, U0, 6, dtype=R.RIPPLE_F64, layout=lay, scheme=R.RIPPLE_RUSANOV1, bc=bc)
           for lay in (R.RIPPLE_SOA, R.RIPPLE_AOS)]
    assert np.array_equal(got[0][0], got[1][0])
    assert_parity(got[0][0], ref, 1e-12, LINF_F64)
    assert got[0][1]["t"] == pytest.approx(info["t"], rel=1e-12)


def test_uniform_state_and_call_split(ctx):
    U0 = inputs.conserved(np.full((40, 50), 0.7), [np.full((40, 50), 0.3), np.full((40, 50), -0.2)],
                          np.full((40, 50), 1.1))
    got, _ = gpu_euler(ctx, U0, 300, dtype=R.RIPPLE_F64, layout=R.RIPPLE_SOA, scheme=R.RIPPLE_RUSANOV1, bc=BCS[0])
    assert np.array_equal(got, U0)
    # more steps than one launch takes, against the same steps in several calls
    U0 = _state((50, 40))
    one, _ = gpu_euler(ctx, U0, 300, dtype=R.RIPPLE_F64, layout=R.RIPPLE_SOA, scheme=R.RIPPLE_RUSANOV1, bc=BCS[1])
    f = R.ripple_field_create(ctx, (50, 40), 4, R.RIPPLE_SOA, 1, R.RIPPLE_F64)
    prm = R.make_fv_params([1.0 / 50, 1.0 / 40], scheme=R.RIPPLE_RUSANOV1, bc=BCS[1])
    R.ripple_field_upload(f, U0)
    for k in (1, 7, 256, 36):
        R.ripple_fv_step(f, prm, k)
    split = R.ripple_field_download(f)
    R.ripple_field_destroy(f)
    assert np.array_equal(one, split)
