"""The FP64 cell sums of the FP32 state against the implicit cell solve in
numpy binary64, from the same inputs and the GPU's own pressure accelerations.

The sums and the solve run in two-float arithmetic (about 2^-44 relative), or
in binary64 where tau/t* or a velocity leaves its range; either way what is
left is the rounding of the cell's results and of the particle update to
binary32: u*', v*' and the two relaxation factors round once (u = 2^-24), the
update has three more roundings, so with one spare
    |v' - v'_ref| <= 8 u (|v| + tau (|A| + |g|) + |u*'|), likewise for dust.
"""
import numpy as np
import pytest

from conftest import gpu_lib

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


def cell_solve(key, nc, tau, g, eps1, gv, acc, moving, du, ts, harmonic, kd):
    N = np.bincount(key[moving], minlength=nc)
    L = np.bincount(kd, minlength=nc)
    has = (N > 0) & (L > 0)
    N1, L1 = np.maximum(N, 1), np.maximum(L, 1)
    mean = lambda v, k, n: np.stack([np.bincount(k, weights=c, minlength=nc) / n for c in v])
    vs, ab = mean(gv[:, moving], key[moving], N1), mean(acc[:, moving], key[moving], N1)
    us = mean(du, kd, L1)
    st = np.where(has, np.bincount(kd, weights=1.0 / ts if harmonic else ts, minlength=nc), 1.0)
    tst = L1 / st if harmonic else st / L1
    eps, rt = eps1 * L1 / N1, tau / tst
    wn = (vs - us + tau * ab) / (1.0 + rt * (1.0 + eps))
    un = us + tau * g[:, None] + rt * wn
    return has, un, un + wn, 1.0 / (1.0 + rt * eps), 1.0 / (1.0 + rt)


# particles per cell from about one (a thread per cell) to dozens; tau/t_stop
# and velocities inside and outside the range of two-float arithmetic
@pytest.mark.parametrize("harmonic", [0, 1])
@pytest.mark.parametrize("tau_over_t,speed", [(20.0, 0.1), (1e9, 0.1), (1e-22, 0.1), (0.5, 1e-28), (0.5, 1e32)])
@pytest.mark.parametrize("dim,n,per_cell", [(1, 700, 40.0), (1, 301, 2.4), (2, 1500, 5.8), (2, 900, 17.0),
                                            (3, 1331, 1.0)])
def test_fp64_cell_sums_of_the_fp32_state(dim, n, per_cell, tau_over_t, speed, harmonic):
    b = gpu_lib()
    rng = np.random.default_rng(dim * 1000 + n)
    side = max(3, int(round((n / per_cell) ** (1.0 / dim))))
    h = 0.24 / side * 2.0 if side >= 8 else 0.1
    f = lambda a: np.asarray(a, np.float32)
    gx, dx = f(rng.uniform(0, 0.999, (dim, n))), f(rng.uniform(0, 0.999, (dim, n)))
    gv, du = f(speed * rng.standard_normal((dim, n))), f(speed * rng.standard_normal((dim, n)))
    tau = 1e-3
    ts = f(tau / tau_over_t * np.exp(rng.uniform(-1, 1, n)))
    frozen = (rng.uniform(size=n) < 0.1).astype(np.uint8)
    g = np.array([0.3, -1.0, 0.2])[:dim] * (speed if speed > 1 else min(1.0, 10 * speed))
    # a sound speed of the order of the velocities keeps the forces in their range
    p = b.make_params(dim, (0.0,) * 3, (1.0,) * 3, (1, 0, 1), h, 1.0 / side, 1.0 / n, 0.3 / n, cs=min(1.0, max(speed, 1e-12)),
                      tstar_mode=harmonic, cell_acc=b.TFSPH_CELL_ACC_FP64)
    with b.Context(p, gx, gv, dx, du, ts, frozen=frozen) as c:
        cells = [int(v) for v in c.info().n_cells][:dim]
        perm_g, key_g = c.debug(b.TFSPH_DEBUG_PERM_G), c.debug(b.TFSPH_DEBUG_KEYS_G)
        perm_d, key_d = c.debug(b.TFSPH_DEBUG_PERM_D), c.debug(b.TFSPH_DEBUG_KEYS_D)
        c.step(tau, tuple(g))
        c.sync()
        acc = c.debug(b.TFSPH_DEBUG_ACC_G).astype(np.float64)
        v1, u1 = c.field(b.TFSPH_FIELD_VEL_G).astype(np.float64), c.field(b.TFSPH_FIELD_VEL_D).astype(np.float64)
    kg, kd = np.empty(n, np.int64), np.empty(n, np.int64)
    kg[perm_g], kd[perm_d] = key_g, key_d
    nc = int(np.prod(cells))
    m = frozen == 0
    # masses as the library holds them (binary32)
    eps1 = float(np.float32(0.3 / n)) / float(np.float32(1.0 / n))
    w = lambda a: a.astype(np.float64)
    has, un, vn, ig, idd = cell_solve(kg, nc, tau, g, eps1, w(gv), acc, m, w(du), w(ts), harmonic, kd)
    assert has.any()
    rg, rd = w(gv) + tau * (acc + g[:, None]), w(du) + tau * g[:, None]
    vr = np.where(has[kg], un[:, kg] + (rg - un[:, kg]) * ig[kg], rg)
    ur = np.where(has[kd], vn[:, kd] + (rd - vn[:, kd]) * idd[kd], rd)
    tiny = 2.0 ** -148  # results below the normal range round to multiples of 2^-149
    bg = 8 * U * (np.abs(w(gv)) + tau * (np.abs(acc) + np.abs(g)[:, None]) + np.abs(un[:, kg])) + tiny
    bd = 8 * U * (np.abs(w(du)) + tau * np.abs(g)[:, None] + np.abs(vn[:, kd])) + tiny
    assert np.all((np.abs(v1 - vr) <= bg)[:, m]), float((np.abs(v1 - vr) / bg)[:, m].max())
    assert np.array_equal(v1[:, ~m], w(gv)[:, ~m])
    assert np.all(np.abs(u1 - ur) <= bd), float((np.abs(u1 - ur) / bd).max())
