"""The binary64 3D pair sums (candidates prefiltered in binary32) where their
tiles are special, against the oracle with the bounds of test_gpu_wide_pairs:
particles on cell faces with 2h just short of a whole number of cells, a box
that does not start at 0 (tiles across its seams keep the periodic image per
pair), and an open axis with wall particles next to the box and, in two
groups, far outside it."""
import numpy as np
import pytest

import workloads
from conftest import gpu_one_step
from parity import check_neighbour_sets, check_one_step

pytestmark = pytest.mark.gpu


def _box(kind, nside, ratio):
    w = workloads.box3d(nside=nside, precision=1, jitter=0.2)
    w.params.update(h=0.5 * ratio / nside)
    if kind == "faces":
        on = np.random.default_rng(4).random(w.gx.shape) < 0.5
        w.gx = np.where(on, np.floor(w.gx * nside) / nside, w.gx)
    elif kind == "offset":
        w.gx, w.dx = w.gx - 0.25, w.dx - 0.25
        w.params.update(lo=(-0.25,) * 3, hi=(0.75,) * 3)
    elif kind == "open":
        w.params.update(periodic=(1, 0, 1))
        lat = (np.stack([a.ravel() for a in np.meshgrid(*[np.arange(nside)] * 3, indexing="ij")]) + 0.5) / nside
        walls = [lat - np.array([[0.0], [s], [0.0]]) for s in (1.0, -1.0)]
        depth = 3.0 / nside
        walls = [a[:, (a[1] > -depth) & (a[1] < 1.0 + depth)] for a in walls]
        # far from the box, neighbours among themselves, in the edge cells all the same
        small = lat[:, (lat < 6.0 / nside).all(0)]
        far = [small + np.array([[0.3], [y], [0.2]]) for y in (1e7, -40.0)]
        extra = np.concatenate(walls + far, axis=1)
        w.frozen = np.concatenate([np.zeros(w.n_gas, np.uint8), np.ones(extra.shape[1], np.uint8)])
        w.gx = np.concatenate([w.gx, extra], axis=1)
        w.gv = np.concatenate([w.gv, np.zeros_like(extra)], axis=1)
    return w


@pytest.mark.parametrize("kind,nside,ratio", [
    ("faces", 24, 1.0 - 2e-6), ("faces", 24, 2.0 - 5e-6), ("faces", 28, 3.0 - 2e-5), ("faces", 12, 2.0 - 5e-6),
    ("offset", 26, 2.4), ("open", 22, 2.4), ("open", 30, 1.7)])
def test_fp64_box(orc, kind, nside, ratio):
    w = _box(kind, nside, ratio)
    gpu = gpu_one_step(w)
    r, errs = check_one_step(orc, w, gpu, 1)
    inv = np.empty_like(r.perm_g)
    inv[r.perm_g] = np.arange(len(r.perm_g))
    check_neighbour_sets(gpu["nb_count"][inv], gpu["nb_fprint"][inv], r)
    print(errs)
    # the far groups and the walls too: densities one by one
    assert np.all(np.abs(gpu["rho_g"] - r.rho_g) <= 1e-12 * r.rho_g)
