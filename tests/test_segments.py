"""The plan-time rule that gives rows with their own mesh to the warp-segment kernels
(csrc/ram_segments.h, compiled here with g++): every ring length of the paper's bump mesh
is taken in both precisions, the positions of a window and of the edges over it fit their
32 bits, and every cell keeps 2^20 units.  CPU only."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

from paper_2305_05362_gb300 import workloads as wl

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2305_05362_gb300", "csrc")
LEAST = 34  # kNsegMinCells
SOURCE = """
#include "ram_segments.h"
extern "C" void fit(const double *x, int n, int least, int f32, int *out)
{
    double *w = new double[n];
    for (int i = 0; i < n; ++i) w[i] = x[i + 1] - x[i];
    ram::NsegFit both[2];
    ram::nseg_fit(x, w, n, least, both);
    const ram::NsegFit f = both[f32 ? 0 : 1];
    delete[] w;
    out[0] = f.cells; out[1] = f.window; out[2] = f.units;
}
"""


@pytest.fixture(scope="module")
def fit(tmp_path_factory):
    d = tmp_path_factory.mktemp("segments")
    (d / "fit.cpp").write_text(SOURCE)
    lib = str(d / "fit.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I", CSRC,
                    str(d / "fit.cpp"), "-o", lib], check=True)
    fn = ctypes.CDLL(lib).fit

    def run(x, f32):
        x = np.ascontiguousarray(x, dtype=np.float64)
        out = (ctypes.c_int * 3)()
        fn(x.ctypes.data_as(ctypes.c_void_p), ctypes.c_int(x.size - 1), ctypes.c_int(LEAST),
           ctypes.c_int(f32), out)
        return list(out)
    return run


def _check(x, cells, window, units):
    n = x.size - 1
    w, L = np.diff(x), x[-1] - x[0]
    assert 1 <= cells <= min(window - 4, n - 1) and window <= 156
    assert cells >= min(60, n - 1)
    xx = np.concatenate([x[:-1], x[:-1] + L, x[:-1] + 2 * L, [x[0] + 3 * L]])

    def longest(c):  # of c consecutive cells
        return np.max(xx[c:c + n] - xx[:n])

    if n > 2 * window:
        span = max(longest(window), longest(cells) + w.max())
        assert math.ldexp(span / L, 64 - units) < 2.0 ** 32
    else:
        assert units >= 32 or math.ldexp(longest(min(window, n)) / L, 64 - units) < 2.0 ** 32
    assert math.ldexp(w.min() / L, 64 - units) >= 2.0 ** 20
    # the source cells that an interval as long as the widest cell touches
    touched = np.searchsorted(xx, xx[:n] + w.max(), side="left") - np.arange(n)
    assert touched.max() + 1 <= window


@pytest.mark.parametrize("first", [256, 400, 508, 640, 800, 1000, 1270, 1530, 2000, 4080, 8190])
def test_bump_mesh_at_every_length(fit, first):
    for n in list(range(first, first + 8)) + [first + 37, first + 101]:
        x = wl.bump_nodes(n, -np.pi, np.pi, 0.1387, 0.2773, 15.0)
        cells, window, units = fit(x, 1)
        assert cells > 0, n
        _check(x, cells, window, units)
        c64, w64, half = fit(x, 0)
        assert c64 > 0 and w64 == 156 and half == 0


@pytest.mark.parametrize("mesh", ["bump", "random", "geometric"])
@pytest.mark.parametrize("n", [34, 64, 77, 100, 152, 163, 200, 319, 700, 5000])
def test_what_is_taken_fits(fit, mesh, n):
    if mesh == "bump":
        x = wl.bump_nodes(n, -np.pi, np.pi, 0.1387, 0.2773, 15.0)
    elif mesh == "random":
        x = wl.random_nodes(n, seed=n)
    else:
        t = np.abs(np.linspace(-1.0, 1.0, n))
        x = np.concatenate([[0.0], np.cumsum(30.0 ** t)]) / np.sum(30.0 ** t)
    cells, window, units = fit(x, 1)
    if cells:
        _check(x, cells, window, units)
    assert fit(x, 0)[0] >= cells


def test_what_is_left(fit):
    """Rows too short, and output cells over more source cells than a window holds."""
    assert fit(wl.random_nodes(33, seed=1), 1)[0] == fit(wl.random_nodes(33, seed=1), 0)[0] == 0
    w = np.ones(600)
    w[300] = 200.0
    x = np.concatenate([[0.0], np.cumsum(w)])
    assert fit(x, 1)[0] == fit(x, 0)[0] == 0
    w[300] = 120.0
    x = np.concatenate([[0.0], np.cumsum(w)])
    assert fit(x, 1)[0] > 0 and fit(x, 0)[0] > 0
