"""Global coordinates that do not fit the idle half of the state at once are
written in parts: crowded binary32 systems, and the smallest ones, against the
same expression evaluated here; and without the cell numbers."""
import ctypes

import numpy as np
import pytest

from paper_1211_1646_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,phi,cells", [
    (4, 4, 0.60, "sigma"),        # 16 disks, 12 to a part
    (8, 8, 0.716, "sqrt2"),
    (331, 350, 0.716, "sqrt2"),
])
def test_positions_in_parts(nx, ny, phi, cells):
    from paper_1211_1646_gb300 import build, hdmc
    build.build()
    Lx, Ly = W.hex_box(nx, ny, phi)
    s = hdmc.System(nx * ny, Lx, Ly, 1.0, 0.1, 4, 3, "fp32", cells=cells)
    s.sweep(7)
    xy, cell = hdmc.hdmc_positions(s.h, s.N)
    only = np.zeros((s.N, 2))
    assert hdmc.lib().hdmc_positions(s.h, only.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), None) == hdmc.HDMC_OK
    loc, cnt = s.state()
    c, j = np.nonzero(np.arange(4)[None, :] < cnt[:, None])
    assert np.array_equal(cell, c)
    w = np.array([s.wx, s.wy]).astype(np.float32).astype(np.float64)
    L = np.array([s.mx, s.my]) * w
    at = np.stack([c % s.mx, c // s.mx], axis=1).astype(np.float64)
    v = s.origin() + (at * w + loc[c, j])
    assert np.array_equal(xy, v - L * np.floor(v / L))
    assert np.array_equal(only, xy)
