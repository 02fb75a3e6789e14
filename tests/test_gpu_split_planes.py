"""Split tiles of the binary64 3D sums: the lanes of a particle share out the
planes of cells the same way whichever walk a lane takes. Particles lie where
the binary32 window of the prefilter is a plane wider than the binary64 one,
beside clusters that overflow the list of one of their lanes only (which then
walks in binary64). Densities one by one against the oracle; bounds of
test_gpu_wide_pairs."""
import numpy as np
import pytest

import workloads
from conftest import gpu_one_step
from parity import check_one_step

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside,cluster", [(18, 90), (20, 120)])
def test_one_lane_without_a_list(orc, nside, cluster):
    w = workloads.box3d(nside=nside, precision=1, jitter=0.1)
    rng = np.random.default_rng(6)
    used = 0
    # clusters a plane above or below the targets, at several places of the box
    for plane in (1, -1):
        for c in ((5, 5, 5), (5, 12, 9), (12, 5, 10), (11, 12, 4)):
            mid = (np.array(c) + np.array([0.5, 0.5, plane + 0.5]))[:, None]
            w.gx[:, used:used + cluster] = (mid + rng.uniform(-0.4, 0.4, (3, cluster))) / nside
            used += cluster
            # 2h is 2.4 cells: with the targets at fraction 0.4 (0.6) of their
            # cell, the third plane down (up) starts at the support's edge
            f = 0.4 + 1e-6 if plane > 0 else 0.6 - 1e-6
            t = (np.array(c)[:, None] + np.stack([rng.uniform(0.2, 0.8, 40), rng.uniform(0.2, 0.8, 40),
                                                  np.full(40, f)])) / nside
            w.gx[:, used:used + 40] = t
            used += 40
    gpu = gpu_one_step(w)
    r, errs = check_one_step(orc, w, gpu, 1)
    assert np.all(np.abs(gpu["rho_g"] - r.rho_g) <= 1e-12 * r.rho_g)
