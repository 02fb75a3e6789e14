"""ISPH and MK on 3D boxes whose tiled cross-phase sums leave targets to a
thread each: tiles that hold far more sources than fit (few targets and many),
layers, and a lattice exactly on the cell faces, which takes no tiles at all.
Against the oracle with the bounds of test_gpu_xdrag, three steps in a row
agreeing with a context of its own each."""
import numpy as np
import pytest

import workloads
from conftest import gpu_lib
from test_gpu_xdrag import _check

pytestmark = pytest.mark.gpu


def _inside(w):
    for x in (w.gx, w.dx):
        x[:] = np.mod(x, 1.0)
        x[x.astype(np.float32) >= 1.0] = 0.0
    return w


def _box(kind):
    rng = np.random.default_rng(9)
    w = workloads.box3d(nside=64 if kind in ("many", "faces") else 46, precision=0, jitter=0.3)
    f = lambda a: np.asarray(a, np.float32).astype(np.float64)
    if kind in ("few", "many"):
        # dust, and some gas, drawn together: tiles of tens of thousands of sources
        for x, n in ((w.dx, 20000), (w.gx, 9000)):
            x[:, :n] = f(0.45 + 0.12 * rng.uniform(size=(3, n)))
    elif kind == "layer":
        w.dx[2] = f(0.3 + np.mod(w.dx[2], 1.0) / 6.0)
    elif kind == "faces":
        n = 64
        lat = np.stack([a.ravel() for a in np.meshgrid(*[np.arange(n)] * 3, indexing="ij")]) / n
        w.gx, w.dx = f(lat), f(lat)
    return _inside(w)


@pytest.mark.parametrize("kind", ["few", "many", "layer", "faces"])
@pytest.mark.parametrize("scheme", [1, 2], ids=["isph", "mk"])
def test_rest_of_the_cross_sums(orc, kind, scheme):
    w = _box(kind)
    if scheme == orc.MK:
        w.tau = 0.5 * float(np.min(w.tstop))
    _check(orc, w, scheme, 0)


@pytest.mark.parametrize("scheme", [1, 2], ids=["isph", "mk"])
def test_a_step_leaves_nothing_for_the_next(scheme):
    """Overflowing tiles, then a state without any, in one context: as in a fresh context."""
    b = gpu_lib()
    ws = [_box("few"), _inside(workloads.box3d(nside=46, precision=0, jitter=0.3))]
    f = lambda a: np.ascontiguousarray(a, np.float32)
    fields = lambda c: [c.field(k) for k in (b.TFSPH_FIELD_POS_G, b.TFSPH_FIELD_VEL_G, b.TFSPH_FIELD_VEL_D)]
    tau = 0.4 * float(min(np.min(w.tstop) for w in ws))
    state = lambda w: [f(a) for a in (w.gx, w.gv, w.dx, w.du, w.tstop)]
    p = b.params_from_dict(ws[0].params, drag=scheme)
    got = []
    with b.Context(p, *state(ws[0])) as c:
        for w in (ws[0], ws[1], ws[0]):
            c.set_state(*state(w))
            c.step(tau, w.g)
            c.step(tau, w.g)
            c.sync()
            got.append(fields(c))
    for w, g in zip((ws[0], ws[1], ws[0]), got):
        with b.Context(p, *state(w)) as c:
            c.step(tau, w.g)
            c.step(tau, w.g)
            c.sync()
            for a, r in zip(g, fields(c)):
                assert np.array_equal(a, r)
