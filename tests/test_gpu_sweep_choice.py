"""A sweep variant that does not exist for a field falls back to the automatic
choice, bit for bit, also where that is a multi-step kernel without a number."""
import numpy as np
import pytest

import inputs
import paper_2104_08571_gb300 as R
from tests.gpu_util import gpu_euler

pytestmark = pytest.mark.gpu
RUS, MH, FORCE = R.RIPPLE_RUSANOV1, R.RIPPLE_MUSCL_HANCOCK_MINMOD, R.RIPPLE_FORCE_SPLIT
CASES = [((130, 70), RUS, R.RIPPLE_F32, 3), ((130, 70), MH, R.RIPPLE_F32, 3), ((130, 70), FORCE, R.RIPPLE_F32, 3),
         ((70, 33, 20), FORCE, R.RIPPLE_F32, 3), ((70, 33, 20), RUS, R.RIPPLE_F32, 3), ((130, 70), RUS, R.RIPPLE_F64, 2),
         ((130, 70), RUS, R.RIPPLE_F64, 3), ((130, 70), MH, R.RIPPLE_F64, 3)]


@pytest.mark.parametrize("dims,scheme,dtype,variant", CASES)
def test_missing_variant_is_the_automatic_choice(dims, scheme, dtype, variant):
    nd = len(dims)
    r = inputs.uniform(sum(dims), (nd + 2) * int(np.prod(dims))).reshape((nd + 2,) + tuple(reversed(dims)))
    U = inputs.conserved(1.0 + 0.3 * r[0], [0.3 * (r[1 + d] - 0.5) for d in range(nd)], 1.0 + 0.3 * r[nd + 1])
    ctx = R.ripple_ctx_create(0)
    try:
        a, _ = gpu_euler(ctx, U, 20, dtype=dtype, scheme=scheme, halo=2)
        b, _ = gpu_euler(ctx, U, 20, dtype=dtype, scheme=scheme, halo=2, variant=variant)
    finally:
        R.ripple_ctx_destroy(ctx)
    assert np.array_equal(a, b)
