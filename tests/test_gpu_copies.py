"""Copies between dense device arrays and fields over the forms they accept: both
layouts on either side, every component count, dense arrays on and off a
16-byte boundary, row lengths that are and are not multiples of 16 bytes, any
halo.  The copies are exact, and write nothing outside the dense array."""
import numpy as np
import pytest

import inputs
import paper_2104_08571_gb300 as R

pytestmark = pytest.mark.gpu
LAYOUTS = (R.RIPPLE_SOA, R.RIPPLE_AOS)


@pytest.fixture(scope="module")
def ctx():
    c = R.ripple_ctx_create(0)
    yield c
    R.ripple_ctx_destroy(c)


@pytest.mark.parametrize("dtype", [R.RIPPLE_F32, R.RIPPLE_F64])
@pytest.mark.parametrize("layout", LAYOUTS)
@pytest.mark.parametrize("dims", [(1, 1), (3, 5), (4, 3), (64, 9), (130, 7), (1, 1, 3), (5, 4, 3), (8, 3, 4)])
def test_device_copies_are_exact(ctx, dtype, layout, dims):
    import torch
    tt = torch.float32 if dtype == R.RIPPLE_F32 else torch.float64
    n = int(np.prod(dims))
    for nc in range(1, 6):
        want = inputs.uniform(n + nc, nc * n).reshape((nc,) + tuple(reversed(dims)))
        want = want.astype(np.float32 if dtype == R.RIPPLE_F32 else np.float64)
        forms = {R.RIPPLE_SOA: want, R.RIPPLE_AOS: np.ascontiguousarray(np.moveaxis(want, 0, -1))}
        for halo in (0, 1, 2, 3, 8):
            f = R.ripple_field_create(ctx, dims, nc, layout, halo, dtype)
            for src_layout in LAYOUTS:
                for off in (0, 1, 4):  # elements from a 16-byte boundary
                    src = torch.zeros(nc * n + 16, dtype=tt, device="cuda")[off:off + nc * n]
                    src.copy_(torch.from_numpy(forms[src_layout].ravel()))
                    torch.cuda.synchronize()
                    R.ripple_field_upload(f, src, src_layout)
                    for dst_layout in LAYOUTS:
                        back = torch.full((nc * n + 16,), -7.0, dtype=tt, device="cuda")
                        torch.cuda.synchronize()
                        R.ripple_field_download(f, dst_layout, out=back[off:off + nc * n])
                        R.ripple_ctx_sync(ctx)
                        got = back.cpu().numpy()
                        assert np.array_equal(got[off:off + nc * n], forms[dst_layout].ravel()), (nc, halo, src_layout, off)
                        assert (got[:off] == -7).all() and (got[off + nc * n:] == -7).all()
            R.ripple_field_destroy(f)
