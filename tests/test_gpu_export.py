"""Global coordinates written by the device against the same expression
evaluated here from the raw state: O + (c w + local), wrapped into the box, in
canonical (cell, slot) order, every binary64 bit."""
import numpy as np
import pytest

from paper_1211_1646_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _wrapped(v, L):
    return v - L * np.floor(v / L)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("nx,ny,phi,cells", [
    (4, 4, 0.60, "sigma"),        # one block of cells, partly filled
    (100, 82, 0.70, "sigma"),     # a ragged last block
    (150, 98, 0.716, "sqrt2"),    # crowded cells: the coordinates exceed the idle buffer in binary32
    (620, 600, 0.70, "sigma"),    # more blocks than one pass of the prefix sum
])
def test_disk_positions(prec, nx, ny, phi, cells):
    from paper_1211_1646_gb300 import build, hdmc
    build.build()
    Lx, Ly = W.hex_box(nx, ny, phi)
    s = hdmc.System(nx * ny, Lx, Ly, 1.0, 0.1, 4, 3, prec, cells=cells)
    s.sweep(7)
    xy, cell = hdmc.hdmc_positions(s.h, s.N)
    loc, cnt = s.state()
    c, j = np.nonzero(np.arange(4)[None, :] < cnt[:, None])
    assert np.array_equal(cell, c)
    w = np.array([s.wx, s.wy]) if prec == "fp64" else np.array([s.wx, s.wy]).astype(np.float32).astype(np.float64)
    L = np.array([Lx, Ly]) if prec == "fp64" else np.array([s.mx, s.my]) * w
    at = np.stack([c % s.mx, c // s.mx], axis=1).astype(np.float64)
    assert np.array_equal(xy, _wrapped(s.origin() + (at * w + loc[c, j]), L))
    s.sweep(3)   # the scratch held nothing that a sweep reads
    t = hdmc.System(nx * ny, Lx, Ly, 1.0, 0.1, 4, 3, prec, cells=cells)
    t.sweep(10)
    assert np.array_equal(s.state()[0], t.state()[0])


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("q,phi", [(8, 0.45), (11, 0.42), (40, 0.49)])
def test_sphere_positions(prec, q, phi):
    from paper_1211_1646_gb300 import build, hdmc
    build.build()
    w3 = W.fcc3(q, phi, 0.1)
    s = hdmc.System3(w3.N, w3.L, 1.0, 0.1, 4, 3, prec)
    s.sweep(7)
    xyz = s.positions()
    loc, cnt = s.state()
    c, j = np.nonzero(np.arange(8)[None, :] < cnt[:, None])
    w = np.asarray(s.w) if prec == "fp64" else np.asarray(s.w).astype(np.float32).astype(np.float64)
    L = np.asarray(s.L) if prec == "fp64" else s.m * w
    at = np.stack([c % s.m[0], c // s.m[0] % s.m[1], c // s.m[0] // s.m[1]], axis=1).astype(np.float64)
    assert np.array_equal(xyz, _wrapped(s.origin() + (at * w + loc[c, j]), L))
    s.sweep(3)
    t = hdmc.System3(w3.N, w3.L, 1.0, 0.1, 4, 3, prec)
    t.sweep(10)
    assert np.array_equal(s.state()[0], t.state()[0])
