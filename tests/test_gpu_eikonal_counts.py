"""Godunov updates counted by an eikonal solve are those performed: in FP64 a
sweep passes over cells none of whose neighbours has changed."""
import numpy as np
import pytest

import paper_2104_08571_gb300 as R

pytestmark = pytest.mark.gpu


def _updates(n, dtype):
    ctx = R.ripple_ctx_create(0)
    try:
        fs = R.ripple_field_create(ctx, (n, 1), 1, R.RIPPLE_SOA, 0, dtype)
        ft = R.ripple_field_create(ctx, (n, 1), 1, R.RIPPLE_SOA, 1, dtype)
        R.ripple_field_upload(fs, np.ones((1, n), np.float64 if dtype == R.RIPPLE_F64 else np.float32))
        st = R.ripple_eikonal_solve(fs, ft, [(0, 0)], 1.0, 1e-6)
        R.ripple_field_destroy(fs)
        R.ripple_field_destroy(ft)
        return st
    finally:
        R.ripple_ctx_destroy(ctx)


@pytest.mark.parametrize("n", [3, 20, 32])
def test_fp64_strip_in_one_tile(n):
    """The front moves a cell a sweep.  The first sweep updates the 32 x 32 cells of the tile; the one after
    cell k has changed updates the cells left and right of it and the one above it (in the tile's row 1)."""
    st = _updates(n, R.RIPPLE_F64)
    assert st["tile_visits"] == 1
    assert st["cell_updates"] == 1024 + sum(3 if k < 31 else 2 for k in range(1, n))


def test_fp32_strip_in_one_tile():
    """Pairs of sweeps over every cell of the tile: 31 to the strip's end, one more that changes nothing."""
    assert _updates(32, R.RIPPLE_F32)["cell_updates"] == 34 * 1024
