"""Batched FP32 steps on packed walks against the direct-staged tiles, bit for
bit, over resident sets that pick short and long walk units (one row to 24),
with sides at the edges of a 60-column strip; and the solo solvers on both
sides of the size where the packed walks take over."""
import numpy as np
import pytest

import inputs
import paper_2104_08571_gb300 as R

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = R.ripple_ctx_create(0)
    yield c
    R.ripple_ctx_destroy(c)


def _run(ctx, states, steps, bc, **cfg):
    R.ripple_batch_configure(ctx, **cfg)
    reqs = [R.euler_request(u, k, [1.0 / u.shape[2], 1.0 / u.shape[1]], bc=bc) for u, k in zip(states, steps)]
    infos = [R.ripple_wait(ctx, t) for t in R.ripple_batch_submit(ctx, reqs)]
    assert all(i["status"] == R.RIPPLE_OK for i in infos)
    return [r["output"] for r in reqs], [i["t"] for i in infos]


SETS = {"one": [(61, 1)], "two": [(60, 5), (59, 64)], "few": [(120, 90), (121, 33), (2, 70), (64, 64)],
        "many": [(48 + i % 15, 40 + i % 7) for i in range(40)], "large": [(500 + i, 300) for i in range(40)]}


@pytest.mark.parametrize("name", sorted(SETS))
@pytest.mark.parametrize("layout", [R.RIPPLE_SOA, R.RIPPLE_AOS])
@pytest.mark.parametrize("bc", [R.RIPPLE_BC_PERIODIC, R.RIPPLE_BC_TRANSMISSIVE])
def test_walks_equal_tiles_bitwise(ctx, name, layout, bc):
    states = [inputs.euler2d_sine(nx, amp=0.1 + 0.01 * (i % 9), ny=ny).astype(np.float32)
              for i, (nx, ny) in enumerate(SETS[name])]
    steps = [3 + i % 4 for i in range(len(states))]
    out = [_run(ctx, states, steps, bc, layout=layout, staging=sg, solo_rounds=False, **more)
           for sg, more in ((1, {}), (2, {}), (0, {}), (2, {"async_queue": True}))]
    for got, t in out[1:]:
        assert t == out[0][1]
        for a, b in zip(got, out[0][0]):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("dims", [(390, 400), (400, 400), (401, 411)])
def test_solo_rounds_equal_batched_bitwise(ctx, dims):
    states = [inputs.euler2d_sine(dims[0], amp=0.2, ny=dims[1]).astype(np.float32)]
    a, ta = _run(ctx, states, [23], R.RIPPLE_BC_PERIODIC, solo_rounds=True)
    b, tb = _run(ctx, states, [23], R.RIPPLE_BC_PERIODIC, solo_rounds=False, staging=1)
    assert ta == tb and np.array_equal(a[0], b[0])
