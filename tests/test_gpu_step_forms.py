"""The step rounds alike whatever came before it: after a density export, with
its phases timed, or as it is (one launch for small contexts, one per phase
otherwise). States are equal bit for bit: adiabatic and viscous gases, axes
that wrap fully, cells much finer than the particles' spacing, and clusters
whose tile does not fit shared memory."""
import numpy as np
import pytest

import workloads
from conftest import gpu_context, gpu_lib

pytestmark = pytest.mark.gpu


def _states(b, w, steps=3):
    out = []
    for form in ("plain", "export", "phases"):
        with gpu_context(w) as c:
            c.profile(form == "phases")
            for _ in range(steps):
                if form == "export":
                    c.field(b.TFSPH_FIELD_RHO_G)
                c.step(w.tau, w.g)
            c.sync()
            fields = [b.TFSPH_FIELD_POS_G, b.TFSPH_FIELD_VEL_G, b.TFSPH_FIELD_POS_D, b.TFSPH_FIELD_VEL_D,
                      b.TFSPH_FIELD_RHO_G] + ([b.TFSPH_FIELD_ENERGY_G] if w.params["eos"] == 1 else [])
            out.append([c.field(f) for f in fields])
    return out


def _same(out):
    for other in out[1:]:
        for a, r in zip(out[0], other):
            assert np.array_equal(a, r)


def _stir(w, speed, seed=1):
    rng = np.random.default_rng(seed)
    w.gv += speed * rng.standard_normal(w.gv.shape) * (1 if w.frozen is None else w.frozen == 0)
    w.du += speed * rng.standard_normal(w.du.shape)
    dt = np.float64 if w.params["precision"] else np.float32
    w.gv, w.du = w.gv.astype(dt).astype(np.float64), w.du.astype(dt).astype(np.float64)
    return w


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("case", ["shock", "shock_large", "viscous_wave", "viscous_column", "adiabatic_box"])
def test_viscous_and_energy_terms(case, prec):
    b = gpu_lib()
    if case.startswith("shock"):
        big = case == "shock_large"
        w = workloads.dustyshock(n_left=17000 if big else 803, n_right=2125 if big else 100, precision=prec)
    elif case == "viscous_wave":
        w = workloads.dustywave(n=1000, precision=prec, amp=1e-2)
        w.params.update(av_alpha=1.0, av_beta=2.0)
    elif case == "viscous_column":
        w = workloads.column2d(nside=40, precision=prec)
        w.params.update(av_alpha=1.0, av_beta=2.0)
    else:
        w = workloads.box3d(nside=12, precision=prec, jitter=0.2)
        w.params.update(av_alpha=1.0, av_beta=2.0, eos=1)
        w.ge = np.linspace(1.0, 2.0, w.n_gas).astype(np.float32).astype(np.float64)
    _same(_states(b, _stir(w, 0.05)))


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("viscous", [False, True])
@pytest.mark.parametrize("case", ["full_y", "full_x", "full_1d", "fine_cells", "cluster_1d", "cluster_2d"])
def test_order_of_the_sums(case, viscous, prec):
    """Random particles, so that the last bits tell one order of a sum from another."""
    b = gpu_lib()
    rng = np.random.default_rng(8)
    dim = 1 if case in ("full_1d", "fine_cells", "cluster_1d") else 2
    n = 900
    x = lambda: rng.uniform(0.0, 0.999, (dim, n))
    h = {"full_y": 0.03, "full_x": 0.03, "full_1d": 0.1, "fine_cells": 0.01, "cluster_1d": 0.004,
         "cluster_2d": 0.02}[case]
    cell = {"full_1d": 0.3, "fine_cells": 1e-4}.get(case, 2.0 * h)
    hi = {"full_y": (1.0, 0.17), "full_x": (0.17, 1.0)}.get(case, (1.0, 1.0))[:dim]
    w = workloads.dustywave(n=n, precision=prec)
    w.gx, w.dx = x(), x()
    if case.startswith("cluster"):
        w.gx = np.concatenate([w.gx, 0.99 + 0.009 * rng.uniform(size=(dim, 6000)), 0.003 * rng.uniform(size=(dim, 3000))],
                              axis=1)
    for k in range(dim):
        w.gx[k] *= hi[k]
        w.dx[k] *= hi[k]
    if prec == 0:
        w.gx, w.dx = (a.astype(np.float32).astype(np.float64) for a in (w.gx, w.dx))
    w.gv, w.du = np.zeros_like(w.gx), np.zeros_like(w.dx)
    w.params.update(dim=dim, periodic=(1,) * dim + (0,) * (3 - dim), hi=hi + (1.0,) * (3 - dim), h=h, cell_size=cell,
                    m_gas=1.0 / n, m_dust=1.0 / n)
    if viscous:
        w.params.update(av_alpha=1.0, av_beta=2.0)
    w.tau = 1e-5
    _same(_states(b, _stir(w, 0.5)))


@pytest.mark.parametrize("cell_acc", [0, 1])
@pytest.mark.parametrize("harmonic", [0, 1])
@pytest.mark.parametrize("case,size,cell,prec", [
    ("wave", 1000, 0.9, 0), ("wave", 1000, 0.9, 1), ("wave", 9000, 1.0, 0), ("wave", 9000, 1.0, 1), ("wave", 60, 1.0, 1),
    ("wave", 4000, 0.4, 0), ("column", 40, 0.8, 0), ("column", 40, 0.8, 1), ("column", 100, 1.0, 0), ("column", 24, 3.0, 1),
    ("wave", 12000, 12.0, 1)])
def test_cells_of_few_and_many_particles(case, size, cell, prec, harmonic, cell_acc):
    """One lane per cell and four give the cell's sums and solve in the same roundings."""
    b = gpu_lib()
    w = workloads.dustywave(n=size, precision=prec, amp=1e-2, cell_factor=cell) if case == "wave" else \
        workloads.column2d(nside=size, precision=prec, cell_factor=cell)
    w.params.update(tstar_mode=harmonic, cell_acc=cell_acc)
    rng = np.random.default_rng(3)
    w.tstop = (w.tstop * np.exp(rng.uniform(-2, 2, w.n_dust))).astype(np.float32).astype(np.float64)
    _same(_states(b, _stir(w, 0.3)))
