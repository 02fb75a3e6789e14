"""The binary64 pair sums of a 3D box large enough for tiles that cross no seam
or one (candidates prefiltered in binary32), against the oracle, with lengths
in units far from 1 (the prefilter works in units of h) and at cells from
about h to several h. Tolerances: parity.check_one_step on the FP64 path."""
import numpy as np
import pytest

import workloads
from conftest import gpu_one_step
from parity import check_neighbour_sets, check_one_step

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("unit", [1.0, 1e-25, 1e25])
@pytest.mark.parametrize("nside,cell_factor", [(26, 1.0), (31, 1.7), (24, 2.9)])
def test_fp64_box(orc, nside, cell_factor, unit):
    w = workloads.box3d(nside=nside, precision=1, jitter=0.2, cell_factor=cell_factor)
    # a pair at the kernel's edge and a coincident pair
    w.gx[:, 1] = w.gx[:, 0] + np.array([2.0 * w.params["h"], 0.0, 0.0])
    w.gx[:, 5] = w.gx[:, 6]
    q = w.params
    w.gx, w.dx = w.gx * unit, w.dx * unit
    q.update(hi=tuple(unit for _ in range(3)), h=q["h"] * unit, cell_size=q["cell_size"] * unit,
             m_gas=q["m_gas"] * unit, m_dust=q["m_dust"] * unit)
    w.tau *= unit
    w.tstop = w.tstop * unit
    gpu = gpu_one_step(w)
    r, errs = check_one_step(orc, w, gpu, 1)
    inv = np.empty_like(r.perm_g)
    inv[r.perm_g] = np.arange(len(r.perm_g))
    check_neighbour_sets(gpu["nb_count"][inv], gpu["nb_fprint"][inv], r)
    print(errs)
