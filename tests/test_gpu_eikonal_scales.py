"""FP32 eikonal solves of one-sided cells: each takes its neighbour's value plus
its own s * h, rounded once, at any scale of s * h (the square of 1e-20 is
below, that of 1e20 above every FP32 number)."""
import numpy as np
import pytest

import inputs
import oracle
import paper_2104_08571_gb300 as R

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = R.ripple_ctx_create(0)
    R.use_torch_allocator(c, 0)
    yield c
    R.ripple_ctx_destroy(c)


def _solve(ctx, s, src, tol):
    dims = tuple(reversed(s.shape))
    fs = R.ripple_field_create(ctx, dims, 1, R.RIPPLE_SOA, 0, R.RIPPLE_F32)
    ft = R.ripple_field_create(ctx, dims, 1, R.RIPPLE_SOA, 1, R.RIPPLE_F32)
    try:
        R.ripple_field_upload(fs, s)
        R.ripple_eikonal_solve(fs, ft, src, 1.0, tol)
        return R.ripple_field_download(ft).reshape(s.shape)
    finally:
        R.ripple_field_destroy(fs)
        R.ripple_field_destroy(ft)


@pytest.mark.parametrize("scale", [1e-30, 1e-20, 1.0, 1e10, 1e20, 1e30])
@pytest.mark.parametrize("dims", [(1, 70), (70, 1), (1, 1, 30), (1, 30, 1), (30, 1, 1)])
def test_strip_is_the_running_sum(ctx, dims, scale):
    """On a strip every cell is one-sided: the running sum of s * h in FP32, bit for bit."""
    n = max(dims)
    s = (np.float32(scale) * (0.5 + 1.5 * inputs.uniform(n + len(dims), n))).astype(np.float32)
    want = np.zeros(n, np.float32)
    for i in range(1, n):
        want[i] = want[i - 1] + s[i]
    T = _solve(ctx, s.reshape(tuple(reversed(dims))), [(0,) * len(dims)], scale * 1e-6)
    assert np.array_equal(T.ravel(), want)


@pytest.mark.parametrize("dims", [(40, 9), (20, 6, 7)])
def test_slow_wall_is_crossed(ctx, dims):
    """A wall two cells thick of slowness 1e20 is slow, not closed: finite times in it and behind it."""
    s = (0.5 + inputs.uniform(5, int(np.prod(dims)))).reshape(tuple(reversed(dims))).astype(np.float32)
    s[..., dims[0] // 2: dims[0] // 2 + 2] = np.float32(1e20)
    src = [tuple(d // 3 for d in dims)]
    T = _solve(ctx, s, src, 1e-6)
    ref = oracle.eikonal_fmm(s.astype(np.float64), 1.0, src)
    assert np.isfinite(T).all()
    # an update rounds to about three units of 6e-8 and a path has under 100 cells; the solve stops at moves below 1e-6
    assert (np.abs(T - ref) <= 2e-5 * ref + 1e-4).all()
