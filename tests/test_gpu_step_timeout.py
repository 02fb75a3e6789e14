"""A one-launch step whose grid barrier may not wait at all gives up and says
so: nothing hangs, steps and exports queued behind it stay in bounds, and a new
state runs as in a fresh context."""
import numpy as np
import pytest

import workloads
from conftest import gpu_context, gpu_lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,prec,after", [(20011, 1, 0), (20011, 1, 2), (30000, 0, 3)])
def test_barrier_timeout_is_reported(n, prec, after):
    b = gpu_lib()
    w = workloads.dustywave(n=n, precision=prec, amp=1e-2)
    dt = np.float64 if prec else np.float32
    fields = lambda c: [c.field(f) for f in (b.TFSPH_FIELD_POS_G, b.TFSPH_FIELD_VEL_G, b.TFSPH_FIELD_POS_D,
                                             b.TFSPH_FIELD_VEL_D)]
    with gpu_context(w) as c:
        for _ in range(after):
            c.step(w.tau, w.g)
        c.sync()
        c.barrier_timeout(0.0)
        c.step(w.tau, w.g)
        c.step(w.tau, w.g)
        c.field(b.TFSPH_FIELD_RHO_G)
        fields(c)
        with pytest.raises(b.TfsphError) as ei:
            c.sync()
        assert ei.value.code == b.TFSPH_E_TIMEOUT
        c.barrier_timeout(2000.0)
        for call in (lambda: c.step(w.tau, w.g), lambda: c.field(b.TFSPH_FIELD_RHO_G), lambda: c.save_state()):
            with pytest.raises(b.TfsphError) as ei:
                call()
            assert ei.value.code == b.TFSPH_E_TIMEOUT
        c.set_state(*[a.astype(dt) for a in (w.gx, w.gv, w.dx, w.du, w.tstop)])
        for _ in range(3):
            c.step(w.tau, w.g)
        c.sync()
        got = fields(c)
        for bad in (-1.0, float("nan")):
            with pytest.raises(b.TfsphError):
                c.barrier_timeout(bad)
    with gpu_context(w) as c:
        for _ in range(3):
            c.step(w.tau, w.g)
        want = fields(c)
    for a, r in zip(got, want):
        assert np.array_equal(a, r)
