"""The batch autotuner returns what runs: for FP32 the steps of TMA staging are
the walks, timed once, so the returned staging does not hang on noise."""
import pytest

import inputs
import paper_2104_08571_gb300 as R

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [R.RIPPLE_F32, R.RIPPLE_F64])
def test_autotune_times_what_runs(dtype):
    ctx = R.ripple_ctx_create(0)
    try:
        cfg, ms = R.ripple_batch_autotune(ctx, [s for s, _ in inputs.batch_problems(24, seed=3)], dtype=dtype)
    finally:
        R.ripple_ctx_destroy(ctx)
    assert all(v > 0 for v in ms.values())
    assert ms[(cfg["layout"], cfg["tile_variant"], cfg["staging"])] == min(ms.values())
    for lay in (R.RIPPLE_SOA, R.RIPPLE_AOS):
        assert ms[(lay, 0, 2)] == ms[(lay, 1, 2)] == ms[(lay, 2, 2)]
        if dtype == R.RIPPLE_F32:
            assert [ms[(lay, v, 0)] for v in range(3)] == [ms[(lay, v, 2)] for v in range(3)]
    if dtype == R.RIPPLE_F32:
        assert cfg["staging"] in (1, 2)
    if cfg["staging"] == 2:
        assert cfg["tile_variant"] == 0
