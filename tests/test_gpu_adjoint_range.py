"""The step's adjoint on the FP32 state where the two-float arithmetic of its
cell sums leaves its exponent range and binary64 takes over (drag, masses,
times, velocities, lambdas far from 1), against the FP64 context on the same
inputs. Tolerance: that of test_gpu_adjoint on the FP32 path, 1e-3 normwise."""
import numpy as np
import pytest

import workloads
from test_gpu_adjoint import _gpu_adjoint

pytestmark = pytest.mark.gpu


# four lanes per cell (the column) and a thread per cell (the box)
@pytest.mark.parametrize("case", ["column", "box"])
@pytest.mark.parametrize("what", ["inside", "drag", "weak_drag", "masses", "times", "velocities", "lambdas"])
def test_adjoint_outside_the_range(case, what):
    w = workloads.column2d(nside=12, precision=0) if case == "column" else workloads.box3d(nside=8, precision=0)
    rng = np.random.default_rng(11)
    f = lambda a: np.asarray(a, np.float32).astype(np.float64)
    moving = np.ones(w.n_gas, bool) if w.frozen is None else w.frozen == 0
    w.gv, w.du = f(0.05 * rng.normal(size=w.gv.shape) * moving), f(0.05 * rng.normal(size=w.du.shape))
    w.tstop = f(w.tau * np.exp(rng.uniform(-1, 1, w.n_dust)))
    scale = 1.0
    if what == "drag":
        w.tstop = f(w.tstop * 2.0 ** -26)
    elif what == "weak_drag":
        w.tstop = f(w.tstop * 2.0 ** 64)
    elif what == "masses":
        w.params["m_dust"] *= 2.0 ** -84  # (the gas's enters cs^2/rho^2 in binary32)
    elif what == "times":
        w.tau, w.tstop = w.tau * 2.0 ** -90, f(w.tstop * 2.0 ** -90)
        w.gv, w.du, w.params["cs"] = w.gv * 2.0 ** 10, w.du * 2.0 ** 10, w.params["cs"] * 2.0 ** 10
        w.g = (0.0, 0.0, 0.0)
    elif what == "velocities":
        w.gv, w.du, w.params["cs"] = w.gv * 2.0 ** -84, w.du * 2.0 ** -84, w.params["cs"] * 2.0 ** -42
        w.g = (0.0, 0.0, 0.0)
    elif what == "lambdas":
        scale = 2.0 ** 64
    lam = [f(scale * rng.normal(size=s)) for s in (w.gx.shape, w.gv.shape, w.dx.shape, w.du.shape)]
    got, ref = _gpu_adjoint(w, lam, precision=0), _gpu_adjoint(w, lam, precision=1)
    for name, a, r in zip(("gx", "gv", "dx", "du", "ts"), got, ref):
        if name in ("gx", "gv"):
            a, r = a[:, moving], r[:, moving]
        s = np.max(np.abs(r))
        assert s < 2.0 ** 120, (name, s)  # a value that binary32 can hold
        assert np.all(np.isfinite(a)), name
        err = np.linalg.norm((a - r) / s) / np.linalg.norm(r / s)
        print(what, name, err)
        assert err < 1e-3, (name, err)
