"""Performance cases of the TFSPH step: what a user's program has the library do.

A pass of the single-context kinds hands a whole particle state over
(``Context.set_state``, device tensors), advances it and exports every field
of the new state in id order, as a program does that couples the step to its
own code. Velocities are O(0.1 c_s) throughout, so that results are not the
rounding residue of a uniform state.

Kinds of case and the sizes they stand for:
  wave      1D periodic dusty sound wave, FP64, 100 + 100 particles and up
  shock     1D dusty shock tube with walls, adiabatic gas with viscosity
  box       3D periodic box with random velocities, 128^3 + 128^3 and below
  column    2D settling column: differentiable rollout with a profile loss
  ensemble  many independent 1D waves stepped as one batch
The 3D box of the implicit cell drag takes one step a pass: over several, a
last-bit difference in a position can move a particle into the next cell,
whose drag is another one.
"""
import math

import numpy as np
import torch

from paper_1908_01682_gb300 import adjoint, binding as b

CFL, H_FACTOR = 0.3, 1.2
DRAG = {"idic": b.TFSPH_DRAG_IDIC, "isph": b.TFSPH_DRAG_ISPH, "mk": b.TFSPH_DRAG_MK}


def listed():
    return [
        # the smallest run: a sound wave of 100 + 100 particles, where launches count
        dict(name="wave_100_fp64", kind="wave", n=100, steps=200),
        # a resolved 1D wave in double precision
        dict(name="wave_20011_fp64", kind="wave", n=20011, steps=20),
        # the dusty shock tube, 2e5 + 2e5 particles: energy equation, viscosity, walls, FP64 cell sums
        dict(name="shock_200000", kind="shock", n=177778, steps=4, cells="fp64"),
        # the headline box, 4.2M particles, as it is in the middle of a run (off the lattice)
        dict(name="box_128_idic", kind="box", n=128, precision="fp32", cells="fp32", drag="idic", jitter=0.3,
             tstar="mean", steps=1),
        # the binding's default options (FP64 cell sums) on an odd grid near its lattice, harmonic mean of t_stop
        dict(name="box_101_fp64_cells", kind="box", n=101, precision="fp32", cells="fp64", drag="idic", jitter=0.05,
             tstar="harmonic", steps=1),
        # a small 3D run: too few tiles to fill the chip
        dict(name="box_24_idic", kind="box", n=24, precision="fp32", cells="fp32", drag="idic", jitter=0.2,
             tstar="mean", steps=1),
        # the paper's two other drag schemes, summed over the particles of the other phase
        dict(name="box_96_isph", kind="box", n=96, precision="fp32", cells="fp32", drag="isph", jitter=0.2,
             tstar="mean", steps=2),
        dict(name="box_75_mk", kind="box", n=75, precision="fp32", cells="fp32", drag="mk", jitter=0.3, tstar="mean",
             steps=2),
        # a 3D box in double precision (reference runs)
        dict(name="box_48_fp64", kind="box", n=48, precision="fp64", cells="fp64", drag="idic", jitter=0.1,
             tstar="mean", steps=1),
        # gradients of a dust-profile loss through a checkpointed rollout of the settling column
        dict(name="column_512_grad", kind="column", n=512, steps=20, every=10, bins=64),
        # the full ensemble: 256 waves of 1k to 64k particles
        dict(name="ensemble_256", kind="ensemble", instances=256, nmin=1024, nmax=65536, steps=10, cells="fp32"),
        # a small ensemble: a few launches' worth of work
        dict(name="ensemble_24", kind="ensemble", instances=24, nmin=128, nmax=4096, steps=20, cells="fp64"),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["wave", "shock", "box", "box", "box", "column", "ensemble", "ensemble"])
    if kind == "wave":
        return dict(kind=kind, n=log_int(64, 30000), steps=rng.randint(10, 60))
    if kind == "shock":
        return dict(kind=kind, n=log_int(4000, 177000), steps=rng.randint(2, 6), cells=rng.choice(["fp32", "fp64"]))
    if kind == "box":
        fp64 = rng.random() < 0.15
        drag = rng.choice(["idic", "idic", "isph", "mk"])
        n = log_int(16, 48) if fp64 else log_int(16, 96 if drag != "idic" else 126)
        return dict(kind=kind, n=n, precision="fp64" if fp64 else "fp32",
                    cells="fp64" if fp64 else rng.choice(["fp32", "fp64"]), drag=drag,
                    jitter=round(rng.uniform(0.05, 0.35), 3), tstar=rng.choice(["mean", "harmonic"]),
                    steps=1 if drag == "idic" else rng.randint(1, 2))
    if kind == "column":
        steps = rng.randint(6, 20)
        return dict(kind=kind, n=log_int(48, 500), steps=steps, every=rng.randint(4, 10), bins=rng.randint(16, 64))
    nmin = log_int(128, 2048)
    return dict(kind=kind, instances=log_int(4, 250), nmin=nmin, nmax=nmin * rng.randint(2, 32),
                steps=rng.randint(4, 12), cells=rng.choice(["fp32", "fp64"]))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(g, shape, lo, hi):
    return lo + (hi - lo) * torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)


def _log_uniform(g, shape, lo, hi):
    return torch.exp(_uniform(g, shape, math.log(lo), math.log(hi)))


def _random_field(g, n, dim, rms):
    """Gaussian random velocity field on n^dim points, |v_k|^2 ~ k^-2, (dim, n^dim), first axis fastest."""
    f = torch.fft.fftfreq(n, device="cuda", dtype=torch.float64) * n
    kk = sum(q * q for q in torch.meshgrid(*([f] * dim), indexing="ij")).sqrt()
    amp = torch.where(kk > 0, 1.0 / kk.clamp(min=1.0), torch.zeros_like(kk))
    v = torch.stack([torch.fft.ifftn(torch.fft.fftn(torch.randn((n,) * dim, generator=g, device="cuda",
                                                                  dtype=torch.float64)) * amp).real.reshape(-1)
                     for _ in range(dim)])
    return v * (rms / (v * v).sum(0).mean().sqrt())


def _lattice(n, dim):
    ax = torch.arange(n, device="cuda", dtype=torch.float64)
    return torch.stack([q.reshape(-1) for q in reversed(torch.meshgrid(*([ax] * dim), indexing="ij"))])


def _wave_arrays(n, amp, phase, shift):
    dx = 1.0 / n
    x0 = (np.arange(n) + 0.5) * dx
    k = 2.0 * math.pi
    xd0 = x0 + shift * dx
    return (np.mod(x0 + amp / k * np.cos(k * x0 + phase), 1.0)[None], amp * np.sin(k * x0 + phase)[None],
            np.mod(xd0 + amp / k * np.cos(k * xd0 + phase), 1.0)[None], amp * np.sin(k * xd0 + phase)[None])


def _inputs(case, seed):
    """(parameters, state as float64 device tensors holding the path's values, tau, g) of the single-context kinds."""
    g = _generator(seed)
    kind, n = case["kind"], case["n"]
    q = dict(eos=0, cs=1.0, gamma=1.4, av_alpha=0.0, av_beta=0.0, tstar_mode=0, lo=(0.0,) * 3, hi=(1.0,) * 3,
             precision=b.TFSPH_FP32, cell_acc=b.TFSPH_CELL_ACC_FP64, drag=b.TFSPH_DRAG_IDIC)
    s = dict(ge=None, frozen=None)
    grav, dxl = (0.0, 0.0, 0.0), 1.0 / n
    h = H_FACTOR * dxl
    if kind == "wave":
        u = _uniform(g, 3, 0.0, 1.0).tolist()
        gx, gv, dx, du = _wave_arrays(n, 1e-4 * (0.5 + u[0]), 2.0 * math.pi * u[1], 0.4 * u[2])
        s.update({k: torch.tensor(v, device="cuda") for k, v in dict(gx=gx, gv=gv, dx=dx, du=du).items()})
        s["ts"] = torch.full((n,), 1e-3, device="cuda", dtype=torch.float64)
        q.update(dim=1, periodic=(1, 0, 0), precision=b.TFSPH_FP64, h=h, cell_size=2.0 * h, m_gas=dxl, m_dust=dxl)
        tau = CFL * h
    elif kind == "shock":
        nl, nr = n, max(1, n // 8)
        dl, dr = 0.5 / nl, 0.5 / nr
        h = H_FACTOR * max(dl, dr)
        ar = lambda m: torch.arange(m, device="cuda", dtype=torch.float64) + 0.5
        xl, xr = ar(nl) * dl, 0.5 + ar(nr) * dr
        wl, wr = -ar(int(math.ceil(2.0 * h / dl)) + 2) * dl, 1.0 + ar(int(math.ceil(2.0 * h / dr)) + 2) * dr
        x = torch.cat([xl, xr, wl, wr])
        left = torch.cat([torch.ones_like(xl), torch.zeros_like(xr), torch.ones_like(wl), torch.zeros_like(wr)])
        rho, p = 0.125 + 0.875 * left, 0.1 + 0.9 * left
        ph = 2.0 * math.pi * _uniform(g, 2, 0.0, 1.0)
        moving = torch.arange(x.numel(), device="cuda") < nl + nr
        # the tube is struck while the gas is in motion
        v = torch.where(moving, 0.1 * torch.sin(2.0 * math.pi * x + ph[0]) * torch.sin(math.pi * x), 0.0 * x)
        xd = torch.cat([xl, xr])
        s.update(gx=x[None], gv=v[None], ge=p / (0.4 * rho), dx=xd[None],
                 du=0.1 * (torch.sin(2.0 * math.pi * xd + ph[1]) * torch.sin(math.pi * xd))[None],
                 ts=_log_uniform(g, nl + nr, 1e-5, 1.0), frozen=(~moving).to(torch.uint8))
        q.update(dim=1, periodic=(0, 0, 0), eos=1, av_alpha=1.0, av_beta=2.0, h=h, cell_size=2.0 * h, m_gas=dl,
                 m_dust=dl)
        tau = CFL * h / math.sqrt(1.4)
    elif kind == "box":
        lat = _lattice(n, 3)
        j = case["jitter"]
        s.update(gx=(lat + 0.25 + _uniform(g, lat.shape, -j, j)) * dxl % 1.0,
                 dx=(lat + 0.75 + _uniform(g, lat.shape, -j, j)) * dxl % 1.0,
                 gv=_random_field(g, n, 3, 0.1), du=_random_field(g, n, 3, 0.1))
        s["ts"] = (torch.full((n ** 3,), 1e-4, device="cuda", dtype=torch.float64) if case["tstar"] == "mean"
                   else _log_uniform(g, n ** 3, 1e-4, 1e-1))
        m = dxl ** 3
        q.update(dim=3, periodic=(1, 1, 1), h=h, cell_size=dxl, m_gas=m, m_dust=m, drag=DRAG[case["drag"]],
                 tstar_mode=int(case["tstar"] == "harmonic"),
                 precision=b.TFSPH_FP64 if case["precision"] == "fp64" else b.TFSPH_FP32)
        # the explicit scheme needs tau < t_stop
        tau = 0.5e-4 if case["drag"] == "mk" else CFL * h / 1.5
    else:  # column
        z = 1.0 - math.exp(-1.0)
        ys = -np.log(1.0 - (np.arange(n) + 0.5) / n * z)
        d0, d1 = ys[1] - ys[0], ys[-1] - ys[-2]
        nw0, nw1 = (int(math.ceil(2.0 * h / d)) + 2 for d in (d0, d1))
        yall = torch.tensor(np.concatenate([ys, ys[0] - (np.arange(nw0) + 1) * d0, ys[-1] + (np.arange(nw1) + 1) * d1]),
                            device="cuda")
        xs = (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) * dxl
        gx = torch.stack([xs.repeat(yall.numel()), yall.repeat_interleave(n)])
        dx = torch.stack([xs.repeat(n), xs.repeat_interleave(n)])
        moving = torch.arange(gx.shape[1], device="cuda") < n * n
        gv = torch.zeros_like(gx)
        # the column is stirred: still at its walls
        gv[:, :n * n] = _random_field(g, n, 2, 0.1) * torch.sin(math.pi * gx[1, :n * n])
        s.update(gx=gx, gv=gv, dx=dx, du=_random_field(g, n, 2, 0.1) * torch.sin(math.pi * dx[1]),
                 ts=_log_uniform(g, n * n, 1e-3, 1e-1), frozen=(~moving).to(torch.uint8))
        q.update(dim=2, periodic=(1, 0, 0), h=h, cell_size=2.0 * h, m_gas=z / (n * n), m_dust=0.01 * z / (n * n))
        tau, grav = CFL * h, (0.0, -1.0, 0.0)
    if case.get("cells") == "fp32":
        q["cell_acc"] = b.TFSPH_CELL_ACC_FP32
    if q["precision"] == b.TFSPH_FP32:
        s = {k: v if v is None or k == "frozen" else v.float().double() for k, v in s.items()}
        for k in ("gx", "dx"):  # a periodic coordinate rounded up to the box edge is its other end
            for d in range(q["dim"]):
                if q["periodic"][d]:
                    s[k][d] = torch.where(s[k][d] >= 1.0, torch.zeros_like(s[k][d]), s[k][d])
    return q, s, tau, grav


def _instances(case, seed):
    """Per instance (parameters, gx, gv, dx, du, t_stop) as numpy float32, and each tau."""
    r = np.random.default_rng(int(seed))
    count = case["instances"]
    # the sizes belong to the case, the waves to the seed
    total = np.exp(np.random.default_rng(5).uniform(math.log(case["nmin"]), math.log(case["nmax"]), count)).astype(int)
    ts = np.exp(r.uniform(math.log(1e-5), 0.0, count))
    amp = np.exp(r.uniform(math.log(2e-2), math.log(1e-1), count))
    phase, shift = r.uniform(0.0, 2.0 * math.pi, count), r.uniform(0.0, 0.4, count)
    out, taus = [], []
    for i in range(count):
        n = max(8, int(total[i]) // 2)
        h = H_FACTOR / n
        q = dict(dim=1, periodic=(1, 0, 0), lo=(0.0,), hi=(1.0,), h=h, cell_size=2.0 * h, m_gas=1.0 / n, m_dust=1.0 / n,
                 cell_acc=b.TFSPH_CELL_ACC_FP32 if case["cells"] == "fp32" else b.TFSPH_CELL_ACC_FP64)
        a = [x.astype(np.float32) for x in _wave_arrays(n, amp[i], phase[i], shift[i])]
        for k in (0, 2):
            a[k][a[k] >= 1.0] = 0.0
        out.append((q, *a, np.full(n, ts[i], np.float32)))
        taus.append(CFL * h)
    return out, taus


# ---------------------------------------------------------------------------
# The passes
# ---------------------------------------------------------------------------
def prepare(case, seed):
    stream = torch.cuda.current_stream()
    if case["kind"] == "ensemble":
        items, taus = _instances(case, seed)
        bt = b.Batch([(b.make_params(**it[0]), *it[1:]) for it in items], stream=stream)
        bt.step(taus, nsteps=0)
        ng, nd = int(bt.goff[-1]), int(bt.doff[-1])
        out = [(f, torch.empty((1, m), device="cuda")) for f, m in
               ((b.TFSPH_FIELD_POS_G, ng), (b.TFSPH_FIELD_VEL_G, ng), (b.TFSPH_FIELD_POS_D, nd),
                (b.TFSPH_FIELD_VEL_D, nd))]
        return dict(kind="ensemble", batch=bt, out=out, steps=case["steps"])
    q, s, tau, grav = _inputs(case, seed)
    dt = torch.float64 if q["precision"] == b.TFSPH_FP64 else torch.float32
    a = {k: v if v is None or k == "frozen" else v.to(dt).contiguous() for k, v in s.items()}
    ctx = b.Context(b.make_params(**q), a["gx"], a["gv"], a["dx"], a["du"], a["ts"], ge=a["ge"], frozen=a["frozen"],
                    stream=stream)
    st = dict(kind=case["kind"], ctx=ctx, a=a, tau=tau, g=grav, steps=case["steps"])
    if case["kind"] == "column":
        grid = adjoint.profile_grid(ctx, (case["bins"], case["bins"]))
        rho0 = adjoint.dust_profile(grid, a["dx"])
        noise = torch.randn(rho0.shape, generator=_generator(seed + 1), device="cuda", dtype=torch.float64)
        st.update(grid=grid, target=rho0 * (1.0 + 0.1 * noise),
                  roll=adjoint.Rollout(ctx, tau, grav, case["steps"], checkpoint_every=case["every"],
                                       frozen=a["frozen"]))
        return st
    fields = [(b.TFSPH_FIELD_POS_G, a["gx"]), (b.TFSPH_FIELD_VEL_G, a["gv"]), (b.TFSPH_FIELD_POS_D, a["dx"]),
              (b.TFSPH_FIELD_VEL_D, a["du"])]
    if a["ge"] is not None:
        fields.append((b.TFSPH_FIELD_ENERGY_G, a["ge"]))
    st["out"] = [(f, torch.empty_like(like)) for f, like in fields]
    return st


def run(st):
    if st["kind"] == "ensemble":
        bt = st["batch"]
        bt.step(nsteps=st["steps"])
        for f, out in st["out"]:
            rc = b.tfsph_batch_fields(bt.b, f, out.data_ptr(), b.TFSPH_MEM_DEVICE)
            if rc != b.TFSPH_OK:
                raise b.TfsphError(rc, b.tfsph_batch_last_error(bt.b))
        return [out for _, out in st["out"]]
    a, ctx = st["a"], st["ctx"]
    if st["kind"] == "column":
        ts, gv, du = (a[k].detach().requires_grad_() for k in ("ts", "gv", "du"))
        gx1, gv1, dx1, du1 = adjoint.TFSPHRollout.apply(ts, gv, du, st["roll"], a["gx"], a["dx"])
        loss = adjoint.DustProfileLoss.apply(dx1, st["target"], st["grid"])
        gts, ggv, gdu = torch.autograd.grad(loss, (ts, gv, du))
        return dict(loss=loss.detach(), grad_ts=gts, grad_gv=ggv, grad_du=gdu, gx=gx1.detach(), gv=gv1.detach(),
                    dx=dx1.detach(), du=du1.detach())
    ctx.set_state(a["gx"], a["gv"], a["dx"], a["du"], a["ts"], ge=a["ge"], frozen=a["frozen"])
    for _ in range(st["steps"]):
        ctx.step(st["tau"], st["g"])
    for f, out in st["out"]:
        ctx.field(f, out=out)
    return [out for _, out in st["out"]]


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
# flops of a pair of particles within 2h: density, pressure force, an ISPH or
# MK cross sum, and the step's adjoint (both transposed pair sums)
FLOPS = dict(density=20, force=35, full_force=70, isph=55, mk=35, adjoint=110)


def work(case):
    kind, steps = case["kind"], case["steps"]
    if kind == "ensemble":
        ratio = case["nmax"] / case["nmin"]
        n = case["instances"] * case["nmin"] * (ratio - 1.0) / math.log(ratio) / 2.0
        # per step: every particle's position, velocity (and t_stop) read and written once
        return dict(bytes=steps * n * (16 + 20) + 4 * n * 4, flops=steps * n * 5 * (FLOPS["density"] + FLOPS["force"]))
    dim = {"wave": 1, "shock": 1, "box": 3, "column": 2}[kind]
    size = 8 if kind == "wave" or case.get("precision") == "fp64" else 4
    n = case["n"] ** dim * (1.125 if kind == "shock" else 1.0)
    near = {"wave": 5.0, "shock": 38.0, "box": 58.0, "column": 18.0}[kind]
    gas, dust = 2 * dim + (kind == "shock"), 2 * dim
    io = n * size * (2 * gas + 2 * dust + 1)                 # the state in and out
    state = n * size * (2 * gas + 2 * dust + 1)              # a step: read and written once
    flops = near * (FLOPS["density"] + FLOPS["full_force" if kind == "shock" else "force"])
    if case.get("drag") == "isph":
        flops += near * (FLOPS["density"] + 2 * FLOPS["isph"])
    elif case.get("drag") == "mk":
        flops += near * 2 * FLOPS["mk"]
    if kind == "column":
        # forward, recomputed forward, and the adjoint step with its four adjoint vectors
        return dict(bytes=3 * io + steps * 4 * state, flops=steps * n * (2 * flops + near * FLOPS["adjoint"]))
    return dict(bytes=io + (steps - 1) * state, flops=steps * n * flops)


# ---------------------------------------------------------------------------
# The same in 64 bits, plain torch
# ---------------------------------------------------------------------------
SIGMA = {1: 2.0 / 3.0, 2: 10.0 / (7.0 * math.pi), 3: 1.0 / math.pi}


def _of(v, i):
    """A per-particle or common quantity at particles i."""
    return v[i] if torch.is_tensor(v) else v


def _pairs(P, tx, sx, off=0):
    """Pairs (target, source) with r < 2h, from a grid of search cells of edge >= 2h. An ensemble's instances lie in
    grids of their own: P["search"] cells per axis, the first one at off, both per particle."""
    dim = tx.shape[0]
    with torch.no_grad():
        lo, ext, ns = [], [], []
        for k in range(dim):
            if P["periodic"][k]:
                lo.append(P["lo"][k])
                ext.append(P["hi"][k] - P["lo"][k])
            else:
                lo.append(min(float(tx[k].min()), float(sx[k].min())))
                ext.append(max(float(tx[k].max()), float(sx[k].max())) - lo[k] + 1e-300)
            ns.append(P["search"] if "search" in P else max(1, int(ext[k] / (2.0 * P["h"]))))
        shared = not torch.is_tensor(ns[0])

        def cells(x):
            c = [((x[k] - lo[k]) * (ns[k] / ext[k])).floor().long().clamp(min=0) for k in range(dim)]
            return [v.clamp(max=n - 1) if shared else torch.minimum(v, n - 1) for v, n in zip(c, ns)]

        def key(c):
            k = c[-1]
            for i in range(dim - 2, -1, -1):
                k = k * ns[i] + c[i]
            return k + off

        tc, sk = cells(tx), key(cells(sx))
        total = int(np.prod(ns)) if shared else P["drag_cells"]
        order = torch.argsort(sk, stable=True)
        count = torch.bincount(sk, minlength=total)
        start = torch.cumsum(count, 0) - count
        ids, A, B = torch.arange(tx.shape[1], device="cuda"), [], []
        few = [n if shared else int(n.min()) for n in ns]
        span = [range(-1, 2) if f >= 3 else range(f) for f in few]  # all cells of an axis of one or two
        for o in np.array(np.meshgrid(*span, indexing="ij")).reshape(dim, -1).T.tolist():
            c, ok = [], torch.ones_like(ids, dtype=torch.bool)
            for k in range(dim):
                v = tc[k] + o[k] if few[k] >= 3 else torch.full_like(ids, o[k])
                if P["periodic"][k]:
                    v = v % ns[k]
                else:
                    ok &= (v >= 0) & (v < ns[k])
                    v = v.clamp(0, ns[k] - 1)
                c.append(v)
            ck = key(c)
            first, have = start[ck], torch.where(ok, count[ck], torch.zeros_like(ck))
            for m in range(int(have.max())):
                a = ids[have > m]
                j = order[first[a] + m]
                r2 = sum(_image(P, k, tx[k][a] - sx[k][j]) ** 2 for k in range(dim))
                keep = r2 < 4.0 * _of(P["h"], a) ** 2
                A.append(a[keep])
                B.append(j[keep])
        return torch.cat(A), torch.cat(B)


def _image(P, k, d):
    if not P["periodic"][k]:
        return d
    L = P["hi"][k] - P["lo"][k]
    return d - L * torch.round(d / L).detach()


def _geometry(P, tx, sx, a, j):
    d = torch.stack([_image(P, k, tx[k][a] - sx[k][j]) for k in range(tx.shape[0])])
    return d, (d * d).sum(0)


def _kernel(P, r2, a, dim, grad=True):
    """W and (1/r) dW/dr (0 at r = 0) of the cubic spline."""
    h = _of(P["h"], a)
    apart = r2.detach() > 0.0
    r = torch.where(apart, r2, torch.ones_like(r2)).sqrt()
    q = torch.where(apart, r / h, torch.zeros_like(r))
    o = (2.0 - q).clamp(min=0.0)
    W = SIGMA[dim] / h ** dim * torch.where(q < 1.0, 1.0 + q * q * (-1.5 + 0.75 * q), 0.25 * o ** 3)
    if not grad:
        return W, None
    g = torch.where(q < 1.0, -3.0 + 2.25 * q, -0.75 * o * o / q.clamp(min=0.5))
    return W, torch.where(apart, SIGMA[dim] / h ** (dim + 2) * g, torch.zeros_like(g))


def _sum(n, a, v):
    return torch.zeros(n, device="cuda", dtype=torch.float64).index_add(0, a, v)


def _keys(P, x, off):
    k = None
    for d in range(x.shape[0] - 1, -1, -1):
        n = P["cells"][d]
        c = ((x[d] - P["lo"][d]) * (n / (P["hi"][d] - P["lo"][d]))).floor().long()
        c = torch.minimum(c.clamp(min=0), n - 1) if torch.is_tensor(n) else c.clamp(0, n - 1)
        k = c if k is None else k * n + c
    return k + off


def _step64(P, s, tau, grav):
    """One step from the state s (float64), Eqs. 17-21 of the paper or its MK / ISPH drag."""
    gx, gv, ge, dx, du, ts = (s[k] for k in ("gx", "gv", "ge", "dx", "du", "ts"))
    dim, ng, nd = gx.shape[0], gx.shape[1], dx.shape[1]
    h, mg, md = P["h"], P["m_gas"], P["m_dust"]
    off = P.get("off", 0)
    a, j = _pairs(P, gx.detach(), gx.detach(), off)
    d, r2 = _geometry(P, gx, gx, a, j)
    W, F = _kernel(P, r2, a, dim)
    rho = mg * _sum(ng, a, W)
    p = P["cs"] ** 2 / rho if ge is None else (P["gamma"] - 1.0) * ge / rho  # p / rho^2
    coef, de = p[a] + p[j], None
    if ge is not None or P["av_alpha"] > 0:
        vr = ((gv[:, a] - gv[:, j]) * d).sum(0)
        mu = torch.where(vr < 0, h * vr / (r2 + 0.01 * h * h), torch.zeros_like(vr))
        c = (P["gamma"] * (P["gamma"] - 1.0) * ge).sqrt() if ge is not None else torch.full_like(rho, P["cs"])
        pi = (-P["av_alpha"] * 0.5 * (c[a] + c[j]) * mu + P["av_beta"] * mu * mu) / (0.5 * (rho[a] + rho[j]))
        coef = coef + pi
        de = mg * _sum(ng, a, (p[a] + 0.5 * pi) * vr * F)
    A = torch.stack([-mg * _sum(ng, a, coef * F * d[k]) for k in range(dim)])
    moving = torch.ones(ng, device="cuda", dtype=torch.bool) if s["frozen"] is None else s["frozen"] == 0
    gvec = torch.tensor(grav[:dim], device="cuda", dtype=torch.float64)[:, None]
    rg, rd = gv + _tau(tau, "gas") * (A + gvec), du + _tau(tau, "dust") * gvec
    if P["drag"] == b.TFSPH_DRAG_IDIC:
        kg, kd = _keys(P, gx.detach(), off), _keys(P, dx.detach(), off)
        nc = P["drag_cells"]
        mv = moving.double()
        N, L = _sum(nc, kg, mv), _sum(nc, kd, torch.ones_like(ts))
        has = (N > 0) & (L > 0)
        N1, L1 = N.clamp(min=1.0), L.clamp(min=1.0)
        mean = lambda v, k, cnt: torch.stack([_sum(nc, k, v[i]) for i in range(dim)]) / cnt
        vs, Ab, us = mean(gv * mv, kg, N1), mean(A * mv, kg, N1), mean(du, kd, L1)
        st = _sum(nc, kd, 1.0 / ts if P["tstar_mode"] else ts)
        st = torch.where(has, st, torch.ones_like(st))
        tstar = L1 / st if P["tstar_mode"] else st / L1
        eps = (L1 / N1 if torch.is_tensor(mg) else md / mg * L1 / N1)  # an ensemble: m_dust = m_gas
        tc = _tau(tau, "cell")
        rt = tc / tstar
        wn = (vs - us + tc * Ab) / (1.0 + rt * (1.0 + eps))
        un = us + tc * gvec + rt * wn
        vn = un + wn
        rg = torch.where(has[kg], un[:, kg] + (rg - un[:, kg]) / (1.0 + rt * eps)[kg], rg)
        rd = torch.where(has[kd], vn[:, kd] + (rd - vn[:, kd]) / (1.0 + rt)[kd], rd)
    else:
        ag, jd = _pairs(P, gx, dx)
        ad, jg = _pairs(P, dx, gx)
        dg, r2g = _geometry(P, gx, dx, ag, jd)
        dd, r2d = _geometry(P, dx, gx, ad, jg)
        Wg, _ = _kernel(P, r2g, ag, dim, False)
        Wd, Fd = _kernel(P, r2d, ad, dim)
        if P["drag"] == b.TFSPH_DRAG_MK:
            e2 = 0.001 * h * h
            fg = ((gv[:, ag] - du[:, jd]) * dg).sum(0) / (r2g + e2) * Wg / ts[jd]
            fd = ((gv[:, jg] - du[:, ad]) * dd).sum(0) / (r2d + e2) * Wd / rho[jg]
            rg = rg + tau * torch.stack([-dim * md / rho * _sum(ng, ag, fg * dg[k]) for k in range(dim)])
            rd = rd + tau * torch.stack([dim * mg / ts * _sum(nd, ad, fd * dd[k]) for k in range(dim)])
        else:
            a2, j2 = _pairs(P, dx, dx)
            rho_d = md * _sum(nd, a2, _kernel(P, _geometry(P, dx, dx, a2, j2)[1], a2, dim, False)[0])
            rdg, K = md * _sum(ng, ag, Wg), md * _sum(ng, ag, Wg / ts[jd])
            ua = torch.stack([md * _sum(ng, ag, Wg * du[k][jd] / rho_d[jd]) for k in range(dim)])
            rgd = mg * _sum(nd, ad, Wd)
            vj = torch.stack([mg * _sum(nd, ad, Wd * gv[k][jg] / rho[jg]) for k in range(dim)])
            qj = P["cs"] ** 2 / rgd
            Aj = -torch.stack([mg * (_sum(nd, ad, p[jg] * Fd * dd[k]) + qj * _sum(nd, ad, Fd * dd[k]))
                               for k in range(dim)])
            al, be = K / rho, K / rdg
            rg = torch.where(rdg > 0, rg - tau * al * (gv - ua + tau * A) / (1.0 + tau * (al + be)), rg)
            al, be = rho_d / (rgd * ts), 1.0 / ts
            rd = torch.where(rgd > 0, rd + tau * be * (vj - du + tau * Aj) / (1.0 + tau * (al + be)), rd)
    gv1 = torch.where(moving, rg, gv)

    def wrap(x):
        return torch.stack([x[k] - (P["hi"][k] - P["lo"][k]) * torch.floor(
            (x[k] - P["lo"][k]) / (P["hi"][k] - P["lo"][k])).detach() if P["periodic"][k] else x[k]
            for k in range(dim)])

    gx1 = torch.where(moving, wrap(gx + _tau(tau, "gas") * gv1), gx)
    return dict(s, gx=gx1, gv=gv1, dx=wrap(dx + _tau(tau, "dust") * rd), du=rd,
                ge=None if ge is None else torch.where(moving, ge + tau * de, ge))


def _tau(tau, what):
    """An ensemble has a tau per particle and per cell."""
    return tau[what] if isinstance(tau, dict) else tau


def _profile64(P, dx, bins):
    """Cloud-in-cell density of the dust on bins x bins (axis 0 fastest): periodic axes wrap, others clamp."""
    f, i = [], []
    for k in range(2):
        t = (dx[k] - P["lo"][k]) / ((P["hi"][k] - P["lo"][k]) / bins) - 0.5
        i.append(t.detach().floor().long())
        f.append(t - i[k])
    rho = torch.zeros(bins * bins, device="cuda", dtype=torch.float64)
    for c in range(4):
        w, at = P["m_dust"] * bins * bins, []
        for k in range(2):
            up = (c >> k) & 1
            w = w * (f[k] if up else 1.0 - f[k])
            v = i[k] + up
            at.append(v % bins if P["periodic"][k] else v.clamp(0, bins - 1))
        rho = rho.index_add(0, at[0] + bins * at[1], w)
    return rho


def exact(case, seed):
    if case["kind"] == "ensemble":
        return _exact_ensemble(case, seed)
    q, s, tau, grav = _inputs(case, seed)
    P = dict(q)
    P["cells"] = [max(1, math.floor((q["hi"][k] - q["lo"][k]) / q["cell_size"])) for k in range(q["dim"])]
    P["drag_cells"] = int(np.prod(P["cells"]))
    if case["kind"] != "column":
        with torch.no_grad():
            for _ in range(case["steps"]):
                s = _step64(P, s, tau, grav)
        return [s[k] for k in ("gx", "gv", "dx", "du")] + ([] if s["ge"] is None else [s["ge"]])
    leaves = {k: s[k].clone().requires_grad_() for k in ("ts", "gv", "du")}
    with torch.no_grad():
        target = _profile64(P, s["dx"], case["bins"])
        noise = torch.randn(target.shape, generator=_generator(seed + 1), device="cuda", dtype=torch.float64)
        target = target * (1.0 + 0.1 * noise)
    names = ("gx", "gv", "dx", "du")

    def one(gx, gv, dx, du, ts):
        t = _step64(P, dict(s, gx=gx, gv=gv, dx=dx, du=du, ts=ts), tau, grav)
        return tuple(t[k] for k in names)

    from torch.utils.checkpoint import checkpoint
    x = (s["gx"], leaves["gv"], s["dx"], leaves["du"])
    for _ in range(case["steps"]):
        x = checkpoint(one, *x, leaves["ts"], use_reentrant=False)
    loss = ((_profile64(P, x[2], case["bins"]) - target) ** 2).sum()
    gts, ggv, gdu = torch.autograd.grad(loss, (leaves["ts"], leaves["gv"], leaves["du"]))
    return dict(loss=loss.detach(), grad_ts=gts, grad_gv=ggv, grad_du=gdu,
                **{k: v.detach() for k, v in zip(names, x)})


def _exact_ensemble(case, seed):
    items, taus = _instances(case, seed)
    dev = lambda v: torch.tensor(np.asarray(v, np.float64), device="cuda")
    n = np.array([it[1].shape[1] for it in items])
    cells = np.array([math.floor(1.0 / it[0]["cell_size"]) for it in items])
    per = lambda v: dev(v).repeat_interleave(torch.tensor(n, device="cuda"))
    first = np.concatenate([[0], np.cumsum(cells)])
    h = per([it[0]["h"] for it in items])
    off, nc = per(first[:-1]).long(), per(cells).long()
    # the drag cells have an edge of 2h or more, so they serve as search cells too
    P = dict(lo=(0.0,), hi=(1.0,), periodic=(1,), h=h, cs=1.0, av_alpha=0.0, tstar_mode=0, drag=b.TFSPH_DRAG_IDIC,
             m_gas=1.0 / per(n), m_dust=1.0 / per(n), cells=[nc], search=nc, drag_cells=int(first[-1]), off=off)
    cat = lambda k: dev(np.concatenate([it[k] for it in items], axis=-1))
    s = dict(gx=cat(1), gv=cat(2), dx=cat(3), du=cat(4), ts=cat(5), ge=None, frozen=None)
    tp = per(taus)
    tau = dict(gas=tp, dust=tp, cell=dev(taus).repeat_interleave(torch.tensor(cells, device="cuda")))
    with torch.no_grad():
        for _ in range(case["steps"]):
            s = _step64(P, s, tau, (0.0, 0.0, 0.0))
    return [s[k] for k in ("gx", "gv", "dx", "du")]
