"""The binning of one position (cell_grid.cuh), compiled for the host: every
finite coordinate, however far from the box, gets a cell of the grid, and one
within 2^50 boxes its exact place."""
import ctypes
import math
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_2107_11311_gb300 import build

WRAPPER = r"""
#include "cell_grid.cuh"
using namespace aenet;
extern "C" void bin_many(int n, const double *x, const double *box, const double *tilt, const int *nc, int *cell,
                         float *u, double *ud, int *finite) {
    Grid g{};
    for (int a = 0; a < 3; ++a) {
        g.nc[a] = nc[a];
        g.box[a] = box[a];
        g.tilt[a] = tilt[a];
        g.h[a] = box[a] / nc[a];
        g.inv_box[a] = 1.0 / box[a];
        g.inv_h[a] = 1.0 / g.h[a];
        g.inv_boxf[a] = (float)g.inv_box[a];
        g.tri = g.tri || tilt[a] != 0.0;
    }
    g.ht[0] = tilt[0] / nc[1];
    g.ht[1] = tilt[1] / nc[2];
    g.ht[2] = tilt[2] / nc[2];
    for (int i = 0; i < n; ++i) {
        bool ok = true;
        cell[i] = bin_position(x[3 * i], x[3 * i + 1], x[3 * i + 2], g, u + 3 * i, ok, ud + 3 * i);
        finite[i] = ok;
    }
}
"""


@pytest.fixture(scope="module")
def binned(tmp_path_factory):
    d = tmp_path_factory.mktemp("binning")
    (d / "wrapper.cu").write_text(WRAPPER)
    so = d / "wrapper.so"
    subprocess.run([build.nvcc(), "-std=c++17", "-O1", "-Xcompiler", "-fPIC", "-shared", "-I" + build.CSRC, "-o", str(so),
                    str(d / "wrapper.cu")], check=True)
    lib = ctypes.CDLL(str(so))

    def run(x, box, nc, tilt=(0.0, 0.0, 0.0)):
        x = np.ascontiguousarray(x, dtype=np.float64)
        n = len(x)
        out = np.zeros(n, np.int32), np.zeros((n, 3), np.float32), np.zeros((n, 3)), np.zeros(n, np.int32)
        args = [x, np.asarray(box, np.float64), np.asarray(tilt, np.float64), np.asarray(nc, np.int32), *out]
        lib.bin_many(n, *[ctypes.c_void_p(a.ctypes.data) for a in args])
        return out

    return run


def _coordinates(L, nc, seed):
    rng = np.random.default_rng(seed)
    x = np.concatenate([rng.uniform(-1, 1, 4000) * 10.0 ** rng.uniform(-320, 308, 4000),
                        rng.uniform(-1, 1, 4000) * 10.0 ** rng.uniform(14, 22, 4000),
                        rng.uniform(-1, 1, 4000) * L * 2.0 ** rng.uniform(-3, 16, 4000)])
    edges = np.array([k * L / nc * s for k in range(4 * nc) for s in (1.0, -1.0)] + [4096 * L, -4096 * L, 4097 * L])
    big = np.finfo(np.float64).max
    return np.concatenate([x, edges, np.nextafter(edges, -np.inf), np.nextafter(edges, np.inf),
                           [0.0, -0.0, 5e-324, -5e-324, big, -big, math.inf, -math.inf, math.nan]])


@pytest.mark.parametrize("L,nc", [(15.6, 2), (6.7, 1), (51.3, 7), (149.2, 22), (0.9, 1), (3.1e4, 1024)])
def test_every_coordinate_gets_a_cell(binned, L, nc):
    x = _coordinates(L, nc, nc)
    for a in range(3):  # each axis on its own, the others at rest
        p = np.full((len(x), 3), 0.3 * L)
        p[:, a] = x
        cell, u, ud, finite = binned(p, [L] * 3, [nc] * 3)
        assert cell.min() >= 0 and cell.max() < nc ** 3
        assert np.array_equal(finite == 1, np.isfinite(x))
        assert np.isfinite(u).all()
        ci = cell // nc ** a % nc
        h = L / nc
        for k in np.flatnonzero(np.isfinite(x) & (np.abs(x) < 2.0 ** 50 * L)):
            # its place in the box, as cell and coordinate, against exact rational arithmetic;
            # the cell-relative coordinate is FP64, off by a few roundings of L (and of the
            # periodic image: x itself has no more digits)
            d = (Fraction(float(x[k])) - Fraction(float(ud[k, a])) - int(ci[k]) * Fraction(h)) / Fraction(L)
            off = abs(d - round(d)) * Fraction(L)
            assert off <= Fraction(8.0 * 2.0 ** -53) * max(Fraction(L), abs(Fraction(float(x[k]))) / 4), (x[k], ci[k], ud[k, a])
            assert -1e-9 * L <= ud[k, a] <= h + 1e-9 * L


@pytest.mark.parametrize("tilt", [(3.0, -2.0, 4.0), (0.0, 0.0, 1e-3), (900.0, -800.0, 700.0)])
def test_every_coordinate_gets_a_cell_of_a_tilted_box(binned, tilt):
    """Finite coordinates whose back substitution overflows among them."""
    box, nc = (14.0, 0.6, 0.5), (2, 1, 1)
    x = _coordinates(14.0, 2, 3)
    rng = np.random.default_rng(4)
    p = np.stack([rng.permutation(x) for _ in range(3)], 1)
    cell, u, ud, finite = binned(p, box, nc, tilt)
    assert cell.min() >= 0 and cell.max() < 2
    assert np.array_equal(finite == 1, np.isfinite(p).all(axis=1))
    assert np.isfinite(u).all()
