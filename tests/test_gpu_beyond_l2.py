"""The binary32 sub-sweep above 2M cells, where some forms load the cells before
they draw the trial directions: every form against the oracle, bit for bit."""
import numpy as np
import pytest

import oracle as O
from paper_1211_1646_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,cells,nsel", [
    (1500, 1400, "sigma", 1),
    (1500, 1400, "sigma", 8),
    (1500, 1400, "sigma", 11),     # run-time n_M
    (2000, 1900, "sqrt2", 4),      # crowded cells
    (2000, 1900, "sqrt2", 8),
    (2000, 1900, "sqrt2", 5),      # crowded, run-time n_M
])
def test_sub_sweep_above_2m_cells(nx, ny, cells, nsel):
    from paper_1211_1646_gb300 import build, hdmc
    build.build()
    O.set_threads(8)
    Lx, Ly = W.hex_box(nx, ny, 0.70)
    g = hdmc.System(nx * ny, Lx, Ly, 1.0, 0.11, nsel, 23, "fp32", cells=cells)
    r = O.System(nx * ny, Lx, Ly, 1.0, 0.11, nsel, 23, O.FP32, cells=O.CELLS_SQRT2 if cells == "sqrt2" else O.CELLS_SIGMA)
    assert g.C > 2000000
    g.sweep(2)
    r.sweep(2)
    O.set_threads(1)
    lg, cg = g.state()
    lr, cr = r.state()
    assert np.array_equal(cg, cr)
    assert np.array_equal(lg, lr)
    assert np.array_equal(g.counters(), r.counters())
