"""A grid-barrier wait of a multi-step field kernel that runs out (the bound on
its polls forced to zero): the call reports RIPPLE_ERR_TIMEOUT, with statistics
at once and without them at the next sync, also when another call was queued
in between; after a new upload the field gives an untouched field's bits."""
import numpy as np
import pytest

import inputs
import paper_2104_08571_gb300 as R

pytestmark = pytest.mark.gpu
CASES = {"rusanov_f32": ((300, 280), R.RIPPLE_RUSANOV1, R.RIPPLE_F32), "mh_f32": ((300, 280), R.RIPPLE_MUSCL_HANCOCK_MINMOD, R.RIPPLE_F32),
         "force_f32": ((300, 280), R.RIPPLE_FORCE_SPLIT, R.RIPPLE_F32), "force3_f32": ((70, 50, 40), R.RIPPLE_FORCE_SPLIT, R.RIPPLE_F32),
         "rusanov_f64": ((300, 280), R.RIPPLE_RUSANOV1, R.RIPPLE_F64)}


@pytest.fixture(scope="module")
def ctx():
    c = R.ripple_ctx_create(0)
    yield c
    R.ripple_ctx_destroy(c)


def _state(dims, dtype):
    nd = len(dims)
    r = inputs.uniform(sum(dims), (nd + 2) * int(np.prod(dims))).reshape((nd + 2,) + tuple(reversed(dims)))
    U = inputs.conserved(1.0 + 0.3 * r[0], [0.3 * (r[1 + d] - 0.5) for d in range(nd)], 1.0 + 0.3 * r[nd + 1])
    return np.ascontiguousarray(U, dtype=np.float32 if dtype == R.RIPPLE_F32 else np.float64)


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("stats", [True, False])
def test_run_out_wait_is_reported_and_leaves_nothing_behind(ctx, monkeypatch, name, stats):
    dims, scheme, dtype = CASES[name]
    U = _state(dims, dtype)
    prm = R.make_fv_params([1.0 / n for n in dims], scheme=scheme)
    fields = [R.ripple_field_create(ctx, dims, len(dims) + 2, R.RIPPLE_SOA, 2, dtype) for _ in range(2)]
    try:
        for f in fields:
            R.ripple_field_upload(f, U)
        monkeypatch.setenv("RIPPLE_GRID_SPIN_LIMIT", "0")
        if stats:
            with pytest.raises(R.RippleError) as ei:
                R.ripple_fv_step(fields[0], prm, 6)
            monkeypatch.delenv("RIPPLE_GRID_SPIN_LIMIT")
        else:
            R.ripple_fv_step(fields[0], prm, 6, stats=False)
            monkeypatch.delenv("RIPPLE_GRID_SPIN_LIMIT")
            R.ripple_fv_step(fields[0], prm, 3, stats=False)  # queued before the error is seen
            with pytest.raises(R.RippleError) as ei:
                R.ripple_ctx_sync(ctx)
        assert ei.value.status == R.RIPPLE_ERR_TIMEOUT
        R.ripple_ctx_sync(ctx)  # reported once
        R.ripple_field_upload(fields[0], U)
        for k in (5, 4):
            a, b = (R.ripple_fv_step(f, prm, k) for f in fields)
            assert a["dt_last"] == b["dt_last"] and a["t"] == b["t"]
        assert np.array_equal(R.ripple_field_download(fields[0]), R.ripple_field_download(fields[1]))
    finally:
        for f in fields:
            R.ripple_field_destroy(f)


def test_run_out_wait_of_a_served_walk(ctx, monkeypatch):
    """A request of the size that the packed walks advance alone: its own failure, the runtime keeps serving."""
    def request():
        return R.euler_request(inputs.euler2d_sine(450, amp=0.2, ny=410).astype(np.float32), 40, [1 / 450, 1 / 410])

    def run(r):
        return R.ripple_wait(ctx, R.ripple_batch_submit(ctx, [r])[0], 60000)["status"]

    R.ripple_batch_configure(ctx)
    first, bad, again = request(), request(), request()
    assert run(first) == R.RIPPLE_OK
    monkeypatch.setenv("RIPPLE_GRID_SPIN_LIMIT", "0")
    assert run(bad) == R.RIPPLE_ERR_TIMEOUT
    monkeypatch.delenv("RIPPLE_GRID_SPIN_LIMIT")
    assert run(again) == R.RIPPLE_OK
    assert np.array_equal(first["output"], again["output"])
