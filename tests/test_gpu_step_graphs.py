"""Graphs of one-launch steps, captured and replayed between ordinary steps and
other calls in every order that keeps the double buffers' parity: always the
state of as many ordinary steps."""
import numpy as np
import pytest

import workloads
from conftest import gpu_context, gpu_lib

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# s: an ordinary step, c: capture of two steps (not run), r: replay, p: a step
# with its phases timed (a launch per phase), e: a density export before a step,
# n: a new state
ORDERS = ["crssr", "scrrsss", "scrssrs", "crpprs", "pcrssr", "cresrs", "crsncrss", "nncrssrs", "crsnnrss"]


@pytest.mark.parametrize("n,prec", [(100, 1), (5000, 1), (3000, 0)])
@pytest.mark.parametrize("order", ORDERS)
def test_replays_between_other_calls(order, n, prec):
    b = gpu_lib()
    w = workloads.dustywave(n=n, precision=prec, amp=1e-2)
    dt = np.float64 if prec else np.float32
    arrays = [a.astype(dt) for a in (w.gx, w.gv, w.dx, w.du, w.tstop)]
    stream = torch.cuda.Stream()
    out = []
    for graphs in (True, False):
        with gpu_context(w) as c:
            c.set_stream(stream)
            g = None
            for k in order:
                if k == "c":
                    if graphs:
                        torch.cuda.synchronize()
                        g = torch.cuda.CUDAGraph()
                        with torch.cuda.graph(g, stream=stream):
                            c.step(w.tau, w.g)
                            c.step(w.tau, w.g)
                elif k == "r":
                    if graphs:
                        with torch.cuda.stream(stream):
                            g.replay()
                    else:
                        c.step(w.tau, w.g)
                        c.step(w.tau, w.g)
                elif k == "p":
                    c.profile(True)
                    c.step(w.tau, w.g)
                    c.profile(False)
                elif k == "n":
                    c.set_state(*arrays)
                else:
                    if k == "e":
                        c.field(b.TFSPH_FIELD_RHO_G)
                    c.step(w.tau, w.g)
            c.sync()
            out.append([c.field(f) for f in (b.TFSPH_FIELD_POS_G, b.TFSPH_FIELD_VEL_G, b.TFSPH_FIELD_POS_D,
                                             b.TFSPH_FIELD_VEL_D)])
            c.set_stream(None)
    for a, r in zip(*out):
        assert np.array_equal(a, r)
