"""The one-launch step on every grid its plan can take: clusters of one to
eight CTAs, the sizes on both sides of the cluster's and the form's limits, and
few gas particles beside many dust particles; bit for bit the
phase-per-launch step."""
import numpy as np
import pytest

import workloads
from conftest import gpu_context, gpu_lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,dust", [(7, 1.0), (20, 1.0), (33, 1.0), (64, 1.0), (80, 1.0), (120, 1.0), (150, 1.0),
                                    (170, 1.0), (200, 1.0), (230, 1.0), (255, 1.0), (500, 1.0), (1024, 1.0),
                                    (1025, 1.0), (40, 20.0), (900, 0.1), (32768, 1.0), (32769, 1.0)])
def test_grids(n, dust, prec):
    b = gpu_lib()
    w = workloads.dustywave(n=n, precision=prec, amp=1e-2)
    m = max(1, int(n * dust))
    if m != n:
        d = workloads.dustywave(n=m, precision=prec, amp=1e-2, dust_shift=0.3)
        w.dx, w.du, w.tstop = d.dx, d.du, d.tstop
        w.params["m_dust"] = 1.0 / m
    out, launches = [], []
    for phases in (False, True):
        with gpu_context(w) as c:
            c.profile(phases)
            before = c.info().launches
            for _ in range(4):
                c.step(w.tau, w.g)
            launches.append(c.info().launches - before)
            c.sync()
            out.append([c.field(f) for f in (b.TFSPH_FIELD_POS_G, b.TFSPH_FIELD_VEL_G, b.TFSPH_FIELD_POS_D,
                                             b.TFSPH_FIELD_VEL_D)])
    if n + m <= 65536:
        assert launches[0] == 4
    assert launches[1] >= 32
    for a, r in zip(*out):
        assert np.array_equal(a, r)
