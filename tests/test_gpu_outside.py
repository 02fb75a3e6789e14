"""Particles that have left the box along an open axis, some of them far and in
groups of neighbours: the second step of a run (no state that holds them is
accepted) against the oracle's step from the state exported after the first,
with the bounds of test_gpu_parity and test_gpu_xdrag. Densities and pressure
accelerations on single-lane and split tiles and in FP64 (whose prefilter
leaves such tiles to binary64), ISPH and MK on their tiled sums. (The IDIC
velocities are left out: the edge cells hold groups whose velocities differ by
orders of magnitude, which the bounds, made of a particle's own, do not count.)"""
import dataclasses

import numpy as np
import pytest

import test_gpu_xdrag
import workloads
from conftest import gpu_context, gpu_lib
from parity import KAPPA_STEP, TOL, UNIT, oracle_step

pytestmark = pytest.mark.gpu


def _second_step(nside, prec, drag):
    b = gpu_lib()
    w = workloads.box3d(nside=nside, precision=prec, jitter=0.1)
    w.params.update(periodic=(1, 0, 1))
    w.tau = 0.4e-4
    w.g = (0.0, 0.0, 0.0)
    dt = np.float64 if prec else np.float32
    # layers at both ends leave together, by a little, by half a box and by many boxes
    for x, v in ((w.gx, w.gv), (w.dx, w.du)):
        for lo, hi, by in ((0.0, 0.08, -0.03), (0.9, 1.0, 0.12), (0.45, 0.5, 2.5), (0.3, 0.36, -300.0)):
            sel = (x[1] >= lo) & (x[1] < hi) & (x[0] < 0.3)
            v[1, sel] = by / w.tau
    w.gv, w.du = w.gv.astype(dt).astype(np.float64), w.du.astype(dt).astype(np.float64)
    # (drag strong enough to keep the phases of a layer together)
    w.tstop = np.full(w.n_dust, 1e-4)
    f = (b.TFSPH_FIELD_POS_G, b.TFSPH_FIELD_VEL_G, b.TFSPH_FIELD_POS_D, b.TFSPH_FIELD_VEL_D)
    with gpu_context(w, drag=drag) as c:
        c.step(w.tau, w.g)
        one = [c.field(k).astype(np.float64) for k in f]
        rho = c.field(b.TFSPH_FIELD_RHO_G).astype(np.float64)
        ts = c.field(b.TFSPH_FIELD_TSTOP_D).astype(np.float64)
        # no velocity carries anything across the box again
        c.step(1e-9, w.g)
        c.sync()
        acc = c.debug(b.TFSPH_DEBUG_ACC_G).astype(np.float64)
        two = [c.field(k).astype(np.float64) for k in f]
    w2 = dataclasses.replace(w, gx=one[0], gv=one[1], dx=one[2], du=one[3], tstop=ts, tau=1e-9)
    assert (one[0][1] > 1.0).sum() > 50 and (one[0][1] < 0.0).sum() > 50
    return w2, two, rho, acc


@pytest.mark.parametrize("nside,prec", [(20, 0), (52, 0), (20, 1), (30, 1)])
def test_gas_sums(orc, nside, prec):
    w, _, rho, acc = _second_step(nside, prec, 0)
    _, _, r, _ = oracle_step(orc, w)
    assert np.all(np.abs(rho - r.rho_g) <= TOL[prec] * r.rho_g)
    assert np.all(np.abs(acc - r.acc_g) <= TOL[prec] * np.abs(r.acc_g) + KAPPA_STEP * UNIT[prec] * r.acc_scale_g)


@pytest.mark.parametrize("scheme", [1, 2], ids=["isph", "mk"])
def test_cross_sums(orc, scheme, monkeypatch):
    w, out, _, _ = _second_step(46, 0, scheme)
    monkeypatch.setattr(test_gpu_xdrag, "_run", lambda *a, **k: out)
    test_gpu_xdrag._check(orc, w, scheme, 0)
