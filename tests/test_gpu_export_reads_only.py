"""Exports between two steps leave the state as it is: the neighbour statistics
of a box whose density pass puts several lanes on a particle (and so adds a
particle's terms in another order than the statistics pass)."""
import numpy as np
import pytest

import workloads
from conftest import gpu_context, gpu_lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside,prec", [(10, 0), (24, 0), (14, 1)])
def test_neighbour_statistics_do_not_change_the_step(nside, prec):
    b = gpu_lib()
    w = workloads.box3d(nside=nside, precision=prec, jitter=0.2)
    out = []
    for export in (False, True):
        with gpu_context(w) as c:
            c.step(w.tau, w.g)
            c.field(b.TFSPH_FIELD_RHO_G)
            if export:
                c.debug(b.TFSPH_DEBUG_NEIGH_COUNT)
                c.debug(b.TFSPH_DEBUG_NEIGH_FPRINT)
            snap = c.save_state(np.zeros(c.state_bytes(), np.uint8))
            c.step(w.tau, w.g)
            out.append([snap, c.field(b.TFSPH_FIELD_VEL_G), c.field(b.TFSPH_FIELD_POS_D)])
    for a, r in zip(*out):
        assert np.array_equal(a, r)
