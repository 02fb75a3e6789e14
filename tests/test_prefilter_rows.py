"""The binary32 prefilter of the binary64 3D density, its own header compiled
for the host: no row leaves the staged halo, whatever cell the rounded estimate
gives (one off the stored one included) and however close 2h is to a whole
number of cells; no neighbour is left out; and a particle far outside the box
is told from those the margins hold for."""
import ctypes as C
import subprocess

import pytest

SRC = r"""
#include <string>
#include <random>
#include "prefilter.cuh"
using namespace tfsph;

static void setup(double ratio, int n, int T, Geo<double> &G, TileCfg &C)
{
    tfsph_params p{};
    p.dim = 3;
    for (int d = 0; d < 3; ++d) { p.hi[d] = 1.0; p.periodic[d] = 1; }
    p.h = 0.5 * ratio / n;
    p.cell_size = 1.0 / n;
    p.m_gas = p.m_dust = 1.0;
    p.cs = 1.0;
    const int nc[3] = {n, n, n};
    Phys<double> Ph;
    make_geo_phys<double>(p, nc, (uint32_t)n * n * n, G, Ph);
    for (int d = 0; d < 3; ++d) { C.T[d] = T; C.H[d] = T + 2 * G.R[d]; }
}

// rows outside the halo, over every place of the estimated cell and fractions on its faces
extern "C" long outside(double ratio, int n, int T)
{
    Geo<double> G;
    TileCfg C{};
    setup(ratio, n, T, G, C);
    const Prefilter P = prefilter_of(G, C);
    const float fs[] = {0.0f, 1e-12f, 0.4f, 1.0f - 0x1p-24f, 1.0f, -2.5f, 3.5f};
    const int hs[] = {G.R[0] - 1, G.R[0], G.R[0] + T - 1, G.R[0] + T};
    const int rows = C.H[1] * C.H[2];
    long bad = 0;
    for (int a = 0; a < 64; ++a)
        for (int b = 0; b < 343; ++b) {
            const int h[3] = {hs[a & 3], hs[(a >> 2) & 3], hs[a >> 4]};
            const float f[3] = {fs[b % 7], fs[b / 7 % 7], fs[b / 49]};
            prefilter_rows(P, G.R, C.H, h, f, 0, 1, [&](int u0, int u1) {
                // [u0, u1) within one row of the halo (u1 may be the row's end)
                const int r = u0 / C.H[0] - (u0 % C.H[0] == 0 && u0 == u1 && u0 > 0 ? 1 : 0);
                if (u0 < 0 || u1 < u0 || u1 > (r + 1) * C.H[0] || r >= rows) ++bad;
            });
        }
    return bad;
}

// neighbours (r < 2h) that no row or the distance test leaves out
extern "C" long missed(double ratio, int n, int T, int pairs)
{
    Geo<double> G;
    TileCfg C{};
    setup(ratio, n, T, G, C);
    const Prefilter P = prefilter_of(G, C);
    std::mt19937_64 rng(17);
    std::uniform_real_distribution<double> U(0.0, 1.0);
    std::normal_distribution<double> N;
    long bad = 0;
    for (int m = 0; m < pairs; ++m) {
        double x[3], y[3], v[3], vv = 0.0;  // in cells, relative to the tile's corner
        int h[3], hy[3];
        float f[3];
        for (int k = 0; k < 3; ++k) { v[k] = N(rng); vv += v[k] * v[k]; }
        // every third at the kernel's edge along an axis
        if (m % 3 == 0) { v[0] = v[1] = v[2] = 0.0; v[m / 3 % 3] = m & 1 ? 1.0 : -1.0; vv = 1.0; }
        const double r = ratio * (m % 2 ? 1.0 - 1e-14 : std::cbrt(U(rng))) / std::sqrt(vv);
        for (int k = 0; k < 3; ++k) {
            const double fr = m % 5 == 0 ? (m % 10 ? 0.0 : 1.0 - 0x1p-53) : U(rng);
            h[k] = (int)(U(rng) * T) + G.R[k];
            f[k] = (float)fr;
            x[k] = h[k] - G.R[k] + fr;
            y[k] = x[k] + r * v[k];
            hy[k] = (int)std::floor(y[k]) + G.R[k];
        }
        float q[2][3];
        for (int k = 0; k < 3; ++k) { q[0][k] = (float)(x[k] * G.w[k] * G.inv_h); q[1][k] = (float)(y[k] * G.w[k] * G.inv_h); }
        bool found = false;
        const int cell = hy[0] + C.H[0] * (hy[1] + C.H[1] * hy[2]);
        prefilter_rows(P, G.R, C.H, h, f, 0, 1, [&](int u0, int u1) { found = found || (cell >= u0 && cell < u1); });
        if (!found || !prefilter_near(P, q[0][0] - q[1][0], q[0][1] - q[1][1], q[0][2] - q[1][2]) ||
            !prefilter_holds(P, q[1][0], q[1][1], q[1][2]))
            ++bad;
    }
    return bad;
}

extern "C" int held(double ratio, int n, int T, double cells)
{
    Geo<double> G;
    TileCfg C{};
    setup(ratio, n, T, G, C);
    const float x = (float)(cells * G.w[0] * G.inv_h);
    return prefilter_holds(prefilter_of(G, C), 0.0f, x, 0.0f) ? 1 : 0;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_1908_01682_gb300 import build
    d = tmp_path_factory.mktemp("prefilter")
    (d / "rows.cu").write_text(SRC)
    out = d / "rows.so"
    subprocess.run([build.nvcc(), "-shared", "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC",
                    f"-I{build.CSRC}", f"-I{build.INCLUDE}", "-cudart", "static", "-o", str(out),
                    str(d / "rows.cu")] + build.ARCH, check=True)
    L = C.CDLL(str(out))
    L.outside.argtypes, L.outside.restype = [C.c_double, C.c_int, C.c_int], C.c_long
    L.missed.argtypes, L.missed.restype = [C.c_double, C.c_int, C.c_int, C.c_int], C.c_long
    L.held.argtypes, L.held.restype = [C.c_double, C.c_int, C.c_int, C.c_double], C.c_int
    return L


# 2h in cells: just short of a whole number (by less than the margins widen it), whole, and in between
RATIOS = [k - d for k in (1, 2, 3) for d in (0.0, 1e-7, 1e-6, 5e-6, 2e-5, 3e-5, 1e-3)] + [0.4, 2.4, 2.9]


@pytest.mark.parametrize("ratio", RATIOS)
@pytest.mark.parametrize("T", [1, 5])
def test_rows_stay_in_the_halo_and_miss_no_neighbour(lib, ratio, T):
    assert lib.outside(ratio, 32, T) == 0
    assert lib.missed(ratio, 32, T, 20000) == 0


def test_far_particles_are_told(lib):
    assert lib.held(2.4, 32, 5, -3.0) and lib.held(2.4, 32, 5, 8.0)
    for cells in (-40.0, 40.0, 1e9, -1e300, float("nan"), float("inf")):
        assert not lib.held(2.4, 32, 5, cells)
