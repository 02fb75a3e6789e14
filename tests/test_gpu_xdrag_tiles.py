"""ISPH and MK on 3D boxes large enough for the tiled cross-phase sums, against
the oracle with the bounds of test_gpu_xdrag: seam-shifted tiles, tiles that
keep the periodic image per pair (lo != 0), an open axis, coarser cells, and a
cluster whose halo does not fit shared memory."""
import numpy as np
import pytest

import workloads
from test_gpu_xdrag import _check

pytestmark = pytest.mark.gpu


def _box(kind):
    # "plain" has more targets than a thread each would fill the chip with: the
    # form of the sums is then chosen by how far the particles are scattered
    w = workloads.box3d(nside=64 if kind in ("plain", "scattered") else 46, precision=0, jitter=0.2,
                        cell_factor=1.45 if kind == "coarse" else 1.0)
    if kind == "scattered":
        rng = np.random.default_rng(5)
        for x in (w.gx, w.dx):
            x[:] = np.mod(x + rng.uniform(-0.4, 0.4, x.shape) / 64, 1.0).astype(np.float32)
            x[x >= 1.0] = 0.0
    elif kind == "offset":
        shift = lambda x: (x - 0.25).astype(np.float32).astype(np.float64)
        w.gx, w.dx = shift(w.gx), shift(w.dx)
        w.params.update(lo=(-0.25,) * 3, hi=(0.75,) * 3)
    elif kind == "open":
        w.params.update(periodic=(1, 0, 1))
    elif kind == "cluster":
        # dust drawn together: one tile holds several thousand particles
        rng = np.random.default_rng(3)
        w.dx[:, :6000] = (0.4 + 0.1 * rng.uniform(size=(3, 6000))).astype(np.float32)
    return w


@pytest.mark.parametrize("kind", ["plain", "scattered", "offset", "open", "coarse", "cluster"])
@pytest.mark.parametrize("scheme", [1, 2], ids=["isph", "mk"])
def test_tiled_cross_sums(orc, kind, scheme):
    w = _box(kind)
    if scheme == orc.MK:
        w.tau = 0.5 * float(np.min(w.tstop))
    _check(orc, w, scheme, 0)
