"""Eikonal solves at the sizes where a tile visit's edges fall (32 x 32 and 8^3
tiles held in registers, four cells per thread): one cell, partial rows and
runs, exactly one and just over one tile, sources on tile edges and corners,
several sources in one tile; against Fast Marching."""
import numpy as np
import pytest

import inputs
import oracle
import paper_2104_08571_gb300 as R
from tests.gpu_util import LINF_EIK, LINF_EIK_F64

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = R.ripple_ctx_create(0)
    R.use_torch_allocator(c, 0)
    yield c
    R.ripple_ctx_destroy(c)


def _solve(ctx, s, src, h, dtype, tol):
    dims = tuple(reversed(s.shape))
    fs = R.ripple_field_create(ctx, dims, 1, R.RIPPLE_SOA, 0, dtype)
    ft = R.ripple_field_create(ctx, dims, 1, R.RIPPLE_SOA, 1, dtype)
    try:
        R.ripple_field_upload(fs, s)
        R.ripple_eikonal_solve(fs, ft, src, h, tol)
        return R.ripple_field_download(ft).reshape(s.shape)
    finally:
        R.ripple_field_destroy(fs)
        R.ripple_field_destroy(ft)


CASES = [((1, 40), [(0, 39)]), ((31, 3), [(30, 2)]), ((32, 32), [(0, 0), (31, 31), (31, 0)]),
         ((33, 33), [(31, 32)]), ((64, 5), [(31, 4), (32, 4)]), ((100, 97), [(31, 32), (63, 64), (96, 0)]),
         ((1, 1, 9), [(0, 0, 7)]), ((33, 33), [(32, 32)]), ((1, 1, 9), [(0, 0, 8)]), ((8, 8, 8), [(7, 7, 7), (0, 0, 0)]), ((9, 7, 17), [(8, 3, 8)]),
         ((16, 5, 12), [(7, 3, 3), (8, 4, 4)]), ((25, 30, 20), [(12, 15, 11), (0, 29, 19)])]


@pytest.mark.parametrize("dims,src", CASES)
@pytest.mark.parametrize("dtype", [R.RIPPLE_F32, R.RIPPLE_F64])
def test_tile_edges_vs_fmm(ctx, dims, src, dtype):
    f32 = dtype == R.RIPPLE_F32
    s = inputs.eikonal_slowness(dims, seed=sum(dims))
    if f32:
        s = s.astype(np.float32)
    h = 1.0 / max(dims)
    T = _solve(ctx, s, src, h, dtype, 1e-6 if f32 else 1e-13)
    ref = oracle.eikonal_fmm(s.astype(np.float64), h, src)
    scale = max(ref.max(), 1e-300)
    assert np.abs(T - ref).max() / scale <= (LINF_EIK if f32 else LINF_EIK_F64)
    for c in src:
        assert T[tuple(reversed(c))] == 0.0
