"""The search reach R covers every row that a walk over staged cells may name:
a particle whose rounded cell estimate lies one cell off the cell it is stored
in looks R - 1 cells further at most, so that its rows stay in the halo of R
cells, also where the pruning radius is just short of a whole number of cells.
The walk's arithmetic is restated here, the geometry is the library's."""
import ctypes as C
import subprocess

import pytest

SRC = r"""
#include <string>
#include "tfsph_internal.cuh"
using namespace tfsph;

// Rows past the halo over particles at cell faces (and a few floats beside
// them) of a grid of n cells on [lo, lo + len), the kernel support at `cells`
// cells; *off counts the particles whose estimate is a cell off.
template <class T> long past(double lo, double len, int n, double cells, long *off)
{
    tfsph_params p{};
    p.dim = 1;
    p.lo[0] = lo;
    p.hi[0] = lo + len;
    const double w = (p.hi[0] - p.lo[0]) / n;
    p.h = 0.5 * cells * w;
    p.cell_size = w;
    p.m_gas = p.m_dust = p.cs = 1.0;
    const int nc[3] = {n, 1, 1};
    Geo<T> G;
    Phys<T> Ph;
    make_geo_phys<T>(p, nc, (uint32_t)n, G, Ph);
    // the square root is an approximation in binary32 (relative error below 2^-22)
    const T up = sizeof(T) == 4 ? T(1.0 + 0x1p-22) : T(1);
    const T t = std::sqrt(G.lim2) * up * G.inv_w[0];
    long bad = 0;
    for (int i = 1; i < n; ++i)
        for (int s = -3; s <= 3; ++s) {
            const long double face = (long double)p.lo[0] + (long double)(p.hi[0] - p.lo[0]) * i / n;
            T x = (T)face;
            for (int k = 0; k < std::abs(s); ++k) x = std::nextafter(x, s < 0 ? T(-1e30) : T(1e30));
            const int exact = (int)std::floor(((long double)x - p.lo[0]) * n / (long double)(p.hi[0] - p.lo[0]));
            volatile T d = x - G.lo[0];
            volatile T tc = d * G.inv_w[0];
            const int est = std::min(n - 1, std::max(0, (int)std::floor((T)tc)));
            const T f = tc - T(est);
            if (est == exact + 1 && ++*off && (int)std::floor((T)(f + t)) > G.R[0] - 1) ++bad;
            if (est == exact - 1 && ++*off && (int)std::floor((T)(t - f + T(1))) > G.R[0] - 1) ++bad;
        }
    return bad;
}
extern "C" long past32(double lo, double len, int n, double cells, long *off) { return past<float>(lo, len, n, cells, off); }
extern "C" long past64(double lo, double len, int n, double cells, long *off) { return past<double>(lo, len, n, cells, off); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_1908_01682_gb300 import build
    d = tmp_path_factory.mktemp("reach")
    (d / "reach.cu").write_text(SRC)
    out = d / "reach.so"
    subprocess.run([build.nvcc(), "-shared", "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC",
                    "-Xcompiler", "-ffp-contract=off", f"-I{build.CSRC}", f"-I{build.INCLUDE}", "-cudart", "static",
                    "-o", str(out), str(d / "reach.cu")] + build.ARCH, check=True)
    L = C.CDLL(str(out))
    for f in (L.past32, L.past64):
        f.argtypes = [C.c_double, C.c_double, C.c_int, C.c_double, C.POINTER(C.c_long)]
        f.restype = C.c_long
    return L


@pytest.mark.parametrize("bits,unit", [(32, 2.0 ** -24), (64, 2.0 ** -53)])
@pytest.mark.parametrize("lo,length", [(0.0, 1.0), (-0.25, 1.0), (0.0, 0.7), (3.0, 10.0)])
def test_rows_of_a_cell_off_stay_in_the_halo(lib, bits, unit, lo, length):
    f = lib.past32 if bits == 32 else lib.past64
    off = C.c_long(0)
    worst = 0
    for n in (11, 12, 24, 43, 100, 333):
        for k in (1, 2, 3):
            # the pruning radius 2h + 8 u span + 32 u h reaches k cells at about this many u short of 2h = k cells
            span = max(abs(lo), abs(lo + length)) + length
            short = 8.0 * span * n / length + 16.0 * k
            for e in range(-60, 61):
                cells = k - unit * (short + e * (n / 20.0 + 2.0))
                worst = max(worst, f(lo, length, n, cells, C.byref(off)))
    assert off.value > 0
    assert worst == 0
