"""The one-launch step of small contexts against the step of one launch per
phase, which timing the phases (``Context.profile``) selects. The sums have the
same terms in the same order, so the states are equal bit for bit; the products
of the viscous and energy terms may be contracted differently in the two
compilations (a last bit of a particle's force now and then): those states
agree to a few roundings of the velocities' magnitude.
"""
import numpy as np
import pytest

import workloads
from conftest import gpu_context, gpu_lib

pytestmark = pytest.mark.gpu


def state(b, w, profile, steps, **over):
    with gpu_context(w, **over) as c:
        c.profile(profile)
        launches = c.info().launches
        for _ in range(steps):
            c.step(w.tau, w.g)
        c.sync()
        launches = c.info().launches - launches
        out = [c.field(f) for f in (b.TFSPH_FIELD_POS_G, b.TFSPH_FIELD_VEL_G, b.TFSPH_FIELD_POS_D,
                                    b.TFSPH_FIELD_VEL_D)]
        if w.params["eos"] == 1:
            out.append(c.field(b.TFSPH_FIELD_ENERGY_G))
        keys = [c.debug(k) for k in (b.TFSPH_DEBUG_PERM_G, b.TFSPH_DEBUG_CSTART_G, b.TFSPH_DEBUG_PERM_D,
                                     b.TFSPH_DEBUG_CSTART_D)]
    return out, keys, launches


SHAPES = [
    ("wave", dict(n=8), 1), ("wave", dict(n=37), 0), ("wave", dict(n=100), 1), ("wave", dict(n=4097), 1),
    ("wave", dict(n=9999), 0), ("wave", dict(n=20011), 1),
    ("shock", dict(n_left=800, n_right=100), 0), ("shock", dict(n_left=17000, n_right=2125), 0),
    ("shock", dict(n_left=800, n_right=100), 1),
    ("column", dict(nside=19), 0), ("column", dict(nside=150), 0), ("column", dict(nside=40), 1),
    ("wave", dict(n=600), 1), ("wave", dict(n=2500), 1), ("wave", dict(n=9000), 1), ("column", dict(nside=160), 1),
]


@pytest.mark.parametrize("cell_acc", [0, 1])
@pytest.mark.parametrize("kind,size,prec", SHAPES)
def test_one_launch_step_matches_the_phases(kind, size, prec, cell_acc):
    b = gpu_lib()
    make = {"wave": workloads.dustywave, "shock": workloads.dustyshock, "column": workloads.column2d}[kind]
    w = make(precision=prec, **size)
    if kind == "wave":
        w.gv *= 100.0  # displacements of the order of the lattice's over the steps
    steps = 3
    got, keys, launches = state(b, w, False, steps, cell_acc=cell_acc)
    ref, rkeys, many = state(b, w, True, steps, cell_acc=cell_acc)
    assert launches == steps and many >= 8 * steps
    for a, r in zip(keys, rkeys):
        assert np.array_equal(a, r)
    u = 2.0 ** -53 if prec else 2.0 ** -24
    for a, r in zip(got, ref):
        if kind != "shock":
            assert np.array_equal(a, r)
        else:
            assert np.abs(a.astype(np.float64) - r).max() <= 16 * u * np.abs(r).max()


@pytest.mark.parametrize("n,prec", [(100, 1), (3000, 0)])
def test_captured_steps_replay(n, prec):
    """A graph of two steps, captured after an uncaptured one and replayed twice, is five steps."""
    torch = pytest.importorskip("torch")
    b = gpu_lib()
    w = workloads.dustywave(n=n, precision=prec, amp=1e-2)
    s = torch.cuda.Stream()
    out = []
    for graph in (True, False):
        with gpu_context(w) as c:
            c.set_stream(s)
            c.step(w.tau, w.g)
            if graph:
                g = torch.cuda.CUDAGraph()
                torch.cuda.synchronize()
                with torch.cuda.graph(g, stream=s):
                    c.step(w.tau, w.g)
                    c.step(w.tau, w.g)
                with torch.cuda.stream(s):
                    g.replay()
                    g.replay()
            else:
                for _ in range(4):
                    c.step(w.tau, w.g)
            c.step(w.tau, w.g)  # and a step after the replays
            c.sync()
            out.append([c.field(f) for f in (b.TFSPH_FIELD_POS_G, b.TFSPH_FIELD_VEL_G, b.TFSPH_FIELD_VEL_D)])
            c.set_stream(None)
    for a, r in zip(*out):
        assert np.array_equal(a, r)
