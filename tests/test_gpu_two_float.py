"""Two-float arithmetic (dfloat.cuh) and the third-order reciprocal square root
of the binary64 3D sums (rsqrt_wide), compiled from their headers and run on
the GPU, against exact rationals: the relative error bounds that the headers
state, with u = 2^-24.
  value + float 2 u^2, value + value 3 u^2, value x value 4 u^2, quotient 15 u^2
  (all of them plus the second-order terms of their proofs, below 1 %)
  1/sqrt(x): the rounding of e (2^-54), of the result (2^-53), a truncation
  below 2^-57, together below 2^-52
Then what the FP64 cell sums must hold beyond binary32 sums: cells of a
thousand particles whose velocities cancel, at a drag that gives every particle
the cell's velocity."""
import ctypes as C
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from conftest import gpu_lib

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
U = 2.0 ** -24

SRC = r"""
#include <string>
#include "dfloat.cuh"
#include "pair.cuh"
using namespace tfsph;
__global__ void k_df(int op, const float *ah, const float *al, const float *bh, const float *bl, float *oh, float *ol, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const df a(ah[i], al[i]), b(bh[i], bl[i]);
    const df o = op == 0 ? a + b.h : (op == 1 ? a + b : (op == 2 ? a - b : (op == 3 ? a * b : a / b)));
    oh[i] = o.h;
    ol[i] = o.l;
}
__global__ void k_rsqrt(const double *x, double *y, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = rsqrt_wide(x[i]);
}
extern "C" int run_df(int op, const float *ah, const float *al, const float *bh, const float *bl, float *oh, float *ol, int n)
{
    k_df<<<(n + 255) / 256, 256>>>(op, ah, al, bh, bl, oh, ol, n);
    return (int)cudaDeviceSynchronize();
}
extern "C" int run_rsqrt(const double *x, double *y, int n)
{
    k_rsqrt<<<(n + 255) / 256, 256>>>(x, y, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_1908_01682_gb300 import build
    d = tmp_path_factory.mktemp("two_float")
    (d / "ops.cu").write_text(SRC)
    out = d / "ops.so"
    flags = [f for f in build.NVCC_FLAGS if f not in ("-Xptxas", "-v")]
    subprocess.run([build.nvcc(), "-shared", "-o", str(out), str(d / "ops.cu")] + flags + ["-cudart", "static"],
                   check=True)
    L = C.CDLL(str(out))
    L.run_df.argtypes = [C.c_int] + [C.c_void_p] * 6 + [C.c_int]
    L.run_rsqrt.argtypes = [C.c_void_p] * 2 + [C.c_int]
    return L


def _values(rng, n, spread):
    h = (rng.choice([-1, 1], n) * rng.uniform(1, 2, n) * 2.0 ** rng.integers(-spread, spread + 1, n)).astype(np.float32)
    ulp = np.spacing(np.abs(h)).astype(np.float64)
    l = (rng.uniform(-0.499, 0.499, n) * ulp).astype(np.float32)
    return h, l


@pytest.mark.parametrize("op,bound", [("+f", 2), ("+", 3), ("-", 3), ("*", 4), ("/", 15)])
@pytest.mark.parametrize("spread", [1, 30])
def test_operations_within_their_bounds(lib, op, bound, spread):
    rng = np.random.default_rng(len(op) + bound + spread)
    n = 4000
    a, b = _values(rng, n, spread), _values(rng, n, spread)
    if op in ("+", "-"):  # a third nearly cancels
        k = n // 3
        s = -1 if op == "+" else 1
        b[0][:k] = s * a[0][:k] * (1 + (rng.integers(-3, 4, k) * 2.0 ** -23).astype(np.float32))
        b[1][:k] = (rng.uniform(-0.49, 0.49, k) * np.spacing(np.abs(b[0][:k]))).astype(np.float32)
    t = lambda x: torch.tensor(x, device="cuda")
    dev = [t(x) for x in (*a, *b)]
    oh, ol = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")
    code = {"+f": 0, "+": 1, "-": 2, "*": 3, "/": 4}[op]
    assert lib.run_df(code, *[x.data_ptr() for x in dev], oh.data_ptr(), ol.data_ptr(), n) == 0
    oh, ol = oh.cpu().numpy(), ol.cpu().numpy()
    worst = 0.0
    for i in range(n):
        x = Fraction(float(a[0][i])) + Fraction(float(a[1][i]))
        y = Fraction(float(b[0][i])) + (0 if op == "+f" else Fraction(float(b[1][i])))
        want = {"+f": x + y, "+": x + y, "-": x - y, "*": x * y, "/": x / y if y else Fraction(0)}[op]
        got = Fraction(float(oh[i])) + Fraction(float(ol[i]))
        if want == 0:
            assert got == 0
        else:
            worst = max(worst, float(abs(got - want) / abs(want)))
        assert abs(float(ol[i])) <= 0.5 * float(np.spacing(np.abs(oh[i])))
    print(op, worst / U ** 2)
    assert worst <= 1.01 * bound * U ** 2


def test_reciprocal_square_root(lib):
    rng = np.random.default_rng(3)
    x = np.concatenate([rng.uniform(1, 4, 6000), rng.uniform(1, 2, 6000) * 2.0 ** rng.integers(-900, 900, 6000),
                        [1.0, 4.0, np.nextafter(1.0, 0), np.nextafter(1.0, 2), 2.0 ** -1000]])
    none = np.array([0.0, 5e-324, 2.0 ** -1030, 2.0 ** -1001])
    dev = torch.tensor(np.concatenate([x, none]), device="cuda")
    out = torch.empty_like(dev)
    assert lib.run_rsqrt(dev.data_ptr(), out.data_ptr(), dev.numel()) == 0
    y = out.cpu().numpy()
    assert np.array_equal(y[len(x):], np.zeros(len(none)))
    worst = 0.0
    for a, r in zip(x, y):
        e = Fraction(float(r)) ** 2 * Fraction(float(a)) - 1  # (1 + d)^2 - 1, d the relative error
        worst = max(worst, abs(float(e)) / 2)
    print(worst * 2.0 ** 53)
    assert worst <= 2.0 ** -52


@pytest.mark.parametrize("dim,harmonic", [(1, 0), (1, 1), (2, 0), (3, 0)])
def test_cell_sums_beyond_binary32(dim, harmonic):
    """Four cells of a thousand particles of each phase. With tau/t* = 2^20 a particle keeps id ~ 1e-6 of its
    velocity and takes v* of its cell, so that
        |u' - u'_ref| <= 4 u |v*| + 4 u id (|u| + |v*|)
    asks the cell's mean (1e-4 of the velocities, which cancel) to one rounding of binary32. The same cells summed in
    binary32 (cell_acc 0) are far outside."""
    b = gpu_lib()
    rng = np.random.default_rng(dim)
    n, cells = 4000, 4
    f = lambda a: np.asarray(a, np.float32)
    # no force: gas far apart along the first axis of a long box is not needed, h is small instead
    hi = (4.0,) + (1.0,) * 2
    gx, dx = f(rng.uniform(0, 0.999, (dim, n))), f(rng.uniform(0, 0.999, (dim, n)))
    gx[0] *= 4.0
    dx[0] *= 4.0
    w = lambda a: a.astype(np.float64)
    half = lambda: (lambda a: np.concatenate([a, -a], axis=1))(f(rng.standard_normal((dim, n // 2))))
    # pairs of opposite velocities in the same cell, and a small mean on top
    gv, du = half(), half()
    gx[:, n // 2:], dx[:, n // 2:] = gx[:, :n // 2], dx[:, :n // 2]
    gv, du = f(w(gv) + 1e-4), f(w(du) - 0.7e-4)
    tau = 1e-3
    ts = f(tau * 2.0 ** -20 * np.exp(rng.uniform(-0.1, 0.1, n)))
    h = 1e-6
    p = lambda acc: b.make_params(dim, (0.0,) * 3, hi, (0, 0, 0), h, 1.0, 1.0 / n, 0.3 / n, cs=1e-15, tstar_mode=harmonic,
                                  cell_acc=acc)
    kg, kd = np.floor(w(gx[0])).astype(int), np.floor(w(dx[0])).astype(int)
    assert len(np.unique(kd)) == cells
    N, L = np.bincount(kg, minlength=cells), np.bincount(kd, minlength=cells)
    mean = lambda v, k, m: np.stack([np.bincount(k, weights=w(c), minlength=cells) / m for c in v])
    vs, us = mean(gv, kg, N), mean(du, kd, L)
    st = np.bincount(kd, weights=1.0 / w(ts) if harmonic else w(ts), minlength=cells)
    rt = tau * st / L if harmonic else tau * L / st
    eps = float(np.float32(0.3 / n)) / float(np.float32(1.0 / n)) * L / N
    wn = (vs - us) / (1.0 + rt * (1.0 + eps))
    vn = us + rt * wn + wn
    idd = 1.0 / (1.0 + rt)
    ref = vn[:, kd] + (w(du) - vn[:, kd]) * idd[kd]
    bound = 4 * U * np.abs(vn[:, kd]) + 4 * U * idd[kd] * (np.abs(w(du)) + np.abs(vn[:, kd]))
    err = {}
    for acc in (b.TFSPH_CELL_ACC_FP64, b.TFSPH_CELL_ACC_FP32):
        with b.Context(p(acc), gx, gv, dx, du, ts) as c:
            c.step(tau, (0.0,) * dim)
            c.sync()
            err[acc] = np.abs(w(c.field(b.TFSPH_FIELD_VEL_D)) - ref) / bound
    print({k: float(v.max()) for k, v in err.items()})
    assert err[b.TFSPH_CELL_ACC_FP64].max() <= 1.0
    assert err[b.TFSPH_CELL_ACC_FP32].max() > 4.0
