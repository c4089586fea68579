"""The binary64 sub-sweep in each of its forms (8, 4, 2 lanes per cell, one
thread per cell; chosen by the number of active cells and how crowded they
are) against the oracle, bit for bit: positions, slot order, counters."""
import numpy as np
import pytest

import oracle as O
from paper_1211_1646_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,phi,cells,nsel,sweeps", [
    (94, 110, 0.68, "sigma", 9, 6),       # 8 lanes, ragged rows, more trials than directions drawn ahead
    (61, 62, 0.72, "sqrt2", 7, 12),       # 8 lanes, crowded cells (up to four disks)
    (233, 254, 0.70, "sigma", 4, 3),      # 4 lanes
    (260, 270, 0.66, "sigma", 17, 2),     # 4 lanes, chunked directions
    (331, 350, 0.70, "sigma", 5, 2),      # 2 lanes
    (401, 420, 0.716, "sqrt2", 12, 2),    # 2 lanes, crowded cells
    (531, 560, 0.70, "sigma", 4, 2),      # one thread, n_M fixed
    (541, 540, 0.70, "sigma", 8, 1),
    (551, 544, 0.60, "sigma", 11, 1),     # one thread, run-time n_M
])
def test_forms_of_the_sub_sweep(nx, ny, phi, cells, nsel, sweeps):
    from paper_1211_1646_gb300 import build, hdmc
    build.build()
    Lx, Ly = W.hex_box(nx, ny, phi)
    g = hdmc.System(nx * ny, Lx, Ly, 1.0, 0.11, nsel, 23, "fp64", cells=cells)
    r = O.System(nx * ny, Lx, Ly, 1.0, 0.11, nsel, 23, O.FP64, cells=O.CELLS_SQRT2 if cells == "sqrt2" else O.CELLS_SIGMA)
    g.sweep(sweeps)
    r.sweep(sweeps)
    lg, cg = g.state()
    lr, cr = r.state()
    assert np.array_equal(cg, cr)
    assert np.array_equal(lg, lr)
    assert np.array_equal(g.counters(), r.counters())
