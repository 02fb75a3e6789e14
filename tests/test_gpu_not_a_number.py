"""A particle whose position is no longer a number is nobody's neighbour: the
one-launch step leaves the others as the phase-per-launch step does."""
import numpy as np
import pytest

import workloads
from conftest import gpu_context, gpu_lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("case,size,prec", [("wave", 60, 1), ("wave", 3000, 1), ("wave", 16000, 1), ("wave", 700, 0),
                                            ("column", 30, 1), ("column", 30, 0)])
def test_one_blown_up_particle(case, size, prec):
    b = gpu_lib()
    w = workloads.dustywave(n=size, precision=prec, amp=1e-3) if case == "wave" else \
        workloads.column2d(nside=size, precision=prec)
    w.gv[0, size // 2] = 2e38 if prec == 0 else 1e308
    out = []
    for phases in (False, True):
        with gpu_context(w) as c:
            c.profile(phases)
            c.step(1e3, w.g)   # its position overflows; the periodic image of that is no number
            for _ in range(3):
                c.step(w.tau, w.g)
            c.sync()
            out.append([c.field(f) for f in (b.TFSPH_FIELD_POS_G, b.TFSPH_FIELD_VEL_G, b.TFSPH_FIELD_RHO_G,
                                             b.TFSPH_FIELD_POS_D, b.TFSPH_FIELD_VEL_D)])
    assert np.isnan(out[0][0]).any()
    for a, r in zip(*out):
        assert np.isfinite(r).mean() > 0.5
        assert np.array_equal(a, r, equal_nan=True)
