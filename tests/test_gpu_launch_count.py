"""The kernels that tfsph_info counts for a step of the ISPH and MK drag: six of
the binning, density and force, ISPH's dust density, a sum and an update per
phase, and behind tiled sums the rest and, beyond a thread per target and chip,
the decision between the forms."""
import numpy as np
import pytest

import workloads
from conftest import gpu_context, gpu_lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scheme", [1, 2], ids=["isph", "mk"])
@pytest.mark.parametrize("nside,extra", [(10, 0), (50, 1), (64, 2)])
def test_launches_of_a_step(nside, extra, scheme):
    gpu_lib()
    w = workloads.box3d(nside=nside, precision=0)
    with gpu_context(w, drag=scheme) as c:
        c.step(1e-6, w.g)
        before = c.info().launches
        c.step(1e-6, w.g)
        c.sync()
        assert c.info().launches - before == 6 + 2 + (scheme == 1) + 2 + 2 + extra
