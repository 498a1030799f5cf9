"""A problem and its twin with x and y exchanged take the same time steps: the
wave-speed sum is a sum of separately rounded products, so it does not depend
on which axis comes first.

The states are uniform, so a step leaves them as they are and the second dt is
formed from them by the step kernel itself; the momenta are small binary
fractions, whose squares add up exactly in either order."""
import numpy as np
import pytest

import inputs
import paper_2104_08571_gb300 as R

pytestmark = pytest.mark.gpu
N = 24
DX = (1.0 / 48.3, 1.0 / 31.7, 1.0 / 29.9)
FV = [("rusanov", 2, None), ("rusanov", 2, 2), ("mh", 2, None), ("mh", 2, 2), ("force", 2, None), ("force", 2, 2),
      ("rusanov", 3, None), ("mh", 3, 2), ("mh", 3, 3), ("force", 3, None), ("force", 3, 2)]
SCHEMES = {"rusanov": R.RIPPLE_RUSANOV1, "mh": R.RIPPLE_MUSCL_HANCOCK_MINMOD, "force": R.RIPPLE_FORCE_SPLIT}


@pytest.fixture(scope="module")
def ctx():
    c = R.ripple_ctx_create(0)
    yield c
    R.ripple_ctx_destroy(c)


def _state(i, dims):
    """State i: density and pressure from (1, 2), momenta k / 16 with |k| < 32."""
    r = inputs.uniform(100 + i, 5)
    m = [np.floor(64 * x - 32) / 16 for x in r[2:2 + len(dims)]]
    q = [1 + r[0]] + m + [2.5 * (1 + r[1]) + 0.5 * sum(x * x for x in m) / (1 + r[0])]
    U = np.empty((len(q),) + tuple(reversed(dims)), np.float32)
    for c, v in enumerate(q):
        U[c] = v
    return U


def _swap(U):
    """x and y exchanged: axes and momenta."""
    V = np.ascontiguousarray(np.swapaxes(U, -1, -2))
    V[[1, 2]] = V[[2, 1]]
    return V


@pytest.mark.parametrize("scheme,nd,variant", FV)
def test_twin_takes_the_same_step(ctx, scheme, nd, variant):
    dims = (13, 9, 6)[:nd]
    for i in range(N):
        U, dt = _state(i, dims), []
        for V, dx in ((U, DX), (_swap(U), (DX[1], DX[0], DX[2]))):
            f = R.ripple_field_create(ctx, tuple(reversed(V.shape[1:])), nd + 2, R.RIPPLE_SOA, 2, R.RIPPLE_F32)
            if variant is not None:
                R.ripple_field_set_sweep(f, variant, 0)
            R.ripple_field_upload(f, V)
            dt.append(R.ripple_fv_step(f, R.make_fv_params(dx[:nd], scheme=SCHEMES[scheme]), 2)["dt_last"])
            assert np.array_equal(R.ripple_field_download(f), V)
            R.ripple_field_destroy(f)
        assert dt[0] == dt[1], f"state {i}"


@pytest.mark.parametrize("cfg", [{"staging": 0}, {"staging": 1}, {"staging": 0, "async_queue": True}, {"solo_rounds": True}])
def test_batched_twin_takes_the_same_step(ctx, cfg):
    R.ripple_batch_configure(ctx, **dict({"solo_rounds": False}, **cfg))
    reqs = []
    for i in range(N):
        U = _state(i, (13, 9))
        reqs += [R.euler_request(U, 2, DX[:2]), R.euler_request(_swap(U), 2, (DX[1], DX[0]))]
    if cfg.get("solo_rounds"):
        t = [R.ripple_wait(ctx, R.ripple_batch_submit(ctx, [r])[0])["t"] for r in reqs]
    else:
        t = [R.ripple_wait(ctx, k)["t"] for k in R.ripple_batch_submit(ctx, reqs)]
    assert t[0::2] == t[1::2]
