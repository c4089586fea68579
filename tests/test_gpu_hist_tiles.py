"""Contact histograms of binary32 systems whose blocks do two tiles of cells,
the last block one (partly filled), against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_1211_1646_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,phi,cells", [
    (701, 700, 0.72, "sigma"),
    (1000, 976, 0.70, "sqrt2"),
])
def test_blocks_of_two_tiles(nx, ny, phi, cells):
    from paper_1211_1646_gb300 import build, hdmc
    build.build()
    Lx, Ly = W.hex_box(nx, ny, phi)
    g = hdmc.System(nx * ny, Lx, Ly, 1.0, 0.08, 4, 7, "fp32", cells=cells)
    r = O.System(nx * ny, Lx, Ly, 1.0, 0.08, 4, 7, O.FP32, cells=O.CELLS_SQRT2 if cells == "sqrt2" else O.CELLS_SIGMA)
    assert g.C > 500000
    g.sweep(6)
    r.sweep(6)
    hist = g.pressure()[2]
    assert hist.sum() > 0
    assert np.array_equal(hist, r.histogram())
