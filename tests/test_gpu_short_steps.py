"""Steps queued one behind the other (a short step may start while the last
CTAs of the one before run) against the same steps in calls of one step, bit
for bit, on grids on both sides of the rule that picks the overlapped launch."""
import numpy as np
import pytest

import inputs
import paper_2104_08571_gb300 as R

pytestmark = pytest.mark.gpu
CASES = [((20, 20, 20), R.RIPPLE_MUSCL_HANCOCK_MINMOD, R.RIPPLE_F32), ((65, 30, 17), R.RIPPLE_MUSCL_HANCOCK_MINMOD, R.RIPPLE_F32),
         ((96, 96, 96), R.RIPPLE_MUSCL_HANCOCK_MINMOD, R.RIPPLE_F32), ((90, 40, 33), R.RIPPLE_RUSANOV1, R.RIPPLE_F32),
         ((33, 9, 12), R.RIPPLE_MUSCL_HANCOCK_MINMOD, R.RIPPLE_F64), ((70, 50), R.RIPPLE_MUSCL_HANCOCK_MINMOD, R.RIPPLE_F64),
         ((70, 50), R.RIPPLE_FORCE_SPLIT, R.RIPPLE_F64), ((300, 300), R.RIPPLE_FORCE_SPLIT, R.RIPPLE_F64)]


@pytest.mark.parametrize("dims,scheme,dtype", CASES)
@pytest.mark.parametrize("layout", [R.RIPPLE_SOA, R.RIPPLE_AOS])
def test_queued_steps_equal_single_calls(dims, scheme, dtype, layout):
    nd = len(dims)
    r = inputs.uniform(sum(dims), (nd + 2) * int(np.prod(dims))).reshape((nd + 2,) + tuple(reversed(dims)))
    U = inputs.conserved(1.0 + 0.3 * r[0], [0.3 * (r[1 + d] - 0.5) for d in range(nd)], 1.0 + 0.3 * r[nd + 1])
    U = U.astype(np.float32 if dtype == R.RIPPLE_F32 else np.float64)
    ctx = R.ripple_ctx_create(0)
    prm = R.make_fv_params([1.0 / n for n in dims], scheme=scheme, bc=R.RIPPLE_BC_PERIODIC)
    out = []
    for calls in ([24], [1] * 24):
        f = R.ripple_field_create(ctx, dims, nd + 2, layout, 2, dtype)
        R.ripple_field_upload(f, U)
        for k in calls:
            R.ripple_fv_step(f, prm, k)
        out.append(R.ripple_field_download(f))
        R.ripple_field_destroy(f)
    R.ripple_ctx_destroy(ctx)
    assert np.array_equal(out[0], out[1])
