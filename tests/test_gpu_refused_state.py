"""A refused set_state leaves the context usable: the next step bins the keys
that are there, and the next valid state is accepted and runs as in a fresh
context."""
import numpy as np
import pytest

import workloads
from conftest import gpu_context, gpu_lib

pytestmark = pytest.mark.gpu


def _fields(b, c):
    return [c.field(f) for f in (b.TFSPH_FIELD_POS_G, b.TFSPH_FIELD_VEL_G, b.TFSPH_FIELD_POS_D, b.TFSPH_FIELD_VEL_D)]


@pytest.mark.parametrize("fault", ["t_stop", "outside", "velocity", "no_dust", "nan_and_no_dust"])
@pytest.mark.parametrize("case", ["wave", "box"])
@pytest.mark.parametrize("device", [False, True])
def test_refused_state(case, fault, device):
    torch = pytest.importorskip("torch")
    b = gpu_lib()
    w = workloads.dustywave(n=700, precision=1, amp=1e-2) if case == "wave" else workloads.box3d(nside=9, precision=1)
    good = [w.gx, w.gv, w.dx, w.du, w.tstop]
    bad = [a.copy() for a in good]
    # the refused state in another order, so that its cells are not those of the state before it
    bad[0], bad[1] = bad[0][:, ::-1].copy(), bad[1][:, ::-1].copy()
    bad[2] = np.mod(bad[2] + 0.37, 1.0)
    if fault == "t_stop":
        bad[4][3] = 0.0
    elif fault == "outside":
        bad[0][0, 5] = 1.5
    elif fault in ("velocity", "nan_and_no_dust"):
        bad[1][0, 7] = np.nan
    put = (lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")) if device else np.ascontiguousarray
    good, bad = [put(a) for a in good], [put(a) for a in bad]
    after = []
    for export in (False, True):
        with gpu_context(w) as c:
            c.step(w.tau, w.g)
            if export:  # binning and density of the state to be replaced are there
                c.field(b.TFSPH_FIELD_RHO_G)
            if "no_dust" in fault:
                gas, dust, fz, mem = c._arrays(*bad, None, None)
                dust[-1] = None
                assert b.tfsph_set_state(c.ctx, gas, dust, fz, mem) == b.TFSPH_E_INVALID_ARG
            else:
                with pytest.raises(b.TfsphError):
                    c.set_state(*bad)
            c.step(w.tau, w.g)
            c.sync()
            after.append(_fields(b, c))
            c.set_state(*good)
            for _ in range(3):
                c.step(w.tau, w.g)
            c.sync()
            got = _fields(b, c)
    for a, r in zip(*after):
        assert np.array_equal(a, r, equal_nan=True)
    with gpu_context(w) as c:
        for _ in range(3):
            c.step(w.tau, w.g)
        want = _fields(b, c)
    for a, r in zip(got, want):
        assert np.array_equal(a, r)
