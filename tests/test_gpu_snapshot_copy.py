"""Device snapshots of every alignment the buffer may have (4 bytes up) and of
odd particle and cell counts, whose parts start off the 16-byte boundaries:
byte for byte the host snapshot, and loaded back they resume the run exactly."""
import numpy as np
import pytest

import workloads
from conftest import gpu_context, gpu_lib

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("offset", [0, 4, 8, 12, 16])
@pytest.mark.parametrize("case,precision", [("wave", 0), ("wave", 1), ("box", 0)])
def test_device_snapshot_equals_host_snapshot(case, precision, offset):
    b = gpu_lib()
    w = workloads.dustywave(n=1237, precision=precision) if case == "wave" else workloads.box3d(nside=15, precision=0)
    with gpu_context(w) as c:
        c.step(w.tau, w.g)
        host = c.save_state(np.zeros(c.state_bytes(), np.uint8))
        pad = torch.full((c.state_bytes() + 64,), 0xA5, dtype=torch.uint8, device="cuda")
        buf = pad[offset:offset + c.state_bytes()]
        c.save_state(buf)
        assert np.array_equal(buf.cpu().numpy(), host)
        assert bool((pad[:offset] == 0xA5).all()) and bool((pad[offset + c.state_bytes():] == 0xA5).all())
        c.step(w.tau, w.g)
        ref = [c.field(f) for f in (b.TFSPH_FIELD_POS_G, b.TFSPH_FIELD_VEL_D)]
        c.load_state(buf)
        assert np.array_equal(c.save_state(np.zeros(c.state_bytes(), np.uint8))[72:], host[72:])
        c.step(w.tau, w.g)
        assert all(np.array_equal(a, c.field(f)) for a, f in zip(ref, (b.TFSPH_FIELD_POS_G, b.TFSPH_FIELD_VEL_D)))
        with pytest.raises(b.TfsphError):
            c.load_state(pad[2:2 + c.state_bytes()])
        c.sync()
