"""3D boxes of few tiles, whose density and force passes put two to eight lanes
on a particle, against the oracle (bounds of test_gpu_parity): sizes for each
number of lanes, ragged tiles, a cluster whose lists overflow, and the force
without a list (after a snapshot is loaded)."""
import numpy as np
import pytest

import workloads
from conftest import gpu_context, gpu_lib
from test_gpu_parity import _compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside", [9, 17, 24, 33, 41, 52])
def test_box(orc, nside):
    _compare(orc, workloads.box3d(nside=nside, precision=0, jitter=0.2))


def test_cluster(orc):
    w = workloads.box3d(nside=20, precision=0)
    rng = np.random.default_rng(2)
    w.gx[:, :400] = (0.5 + 0.04 * rng.uniform(size=(3, 400))).astype(np.float32)
    _compare(orc, w)


def test_force_without_a_list():
    b = gpu_lib()
    w = workloads.box3d(nside=24, precision=0, jitter=0.2)
    with gpu_context(w) as c:
        snap = c.save_state(np.zeros(c.state_bytes(), np.uint8))  # with its forces, from the list
        acc = c.debug(b.TFSPH_DEBUG_ACC_G).astype(np.float64)
        c.load_state(snap)
        c.step(1e-30, w.g)   # leaves the positions where they are
        c.step(1e-30, w.g)
        again = c.debug(b.TFSPH_DEBUG_ACC_G).astype(np.float64)
    # the same terms, added lane by lane in either case
    assert np.array_equal(acc, again)
