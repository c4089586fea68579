"""Contact histograms against the oracle where the scan of half the
neighbourhood can go wrong: grids of four cells per axis (both sides of a cell
are the same cell), ragged rows, more than one tile per block, wide and crowded
cells."""
import numpy as np
import pytest

import oracle as O
from paper_1211_1646_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PREC = {"fp64": O.FP64, "fp32": O.FP32}


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("nx,ny,phi,cells", [
    (4, 4, 0.66, "sigma"),
    (5, 62, 0.723, "sigma"),      # four columns of wide cells
    (70, 62, 0.74, "sigma"),
    (170, 180, 0.72, "sigma"),    # several tiles per block, the last one partly filled
    (150, 98, 0.716, "sqrt2"),
])
def test_histogram_equals_the_oracles(prec, nx, ny, phi, cells):
    from paper_1211_1646_gb300 import build, hdmc
    build.build()
    Lx, Ly = W.hex_box(nx, ny, phi)
    oc = O.CELLS_SQRT2 if cells == "sqrt2" else O.CELLS_SIGMA
    g = hdmc.System(nx * ny, Lx, Ly, 1.0, 0.08, 4, 7, prec, cells=cells)
    r = O.System(nx * ny, Lx, Ly, 1.0, 0.08, 4, 7, PREC[prec], cells=oc)
    seen = 0
    for _ in range(4):
        g.sweep(8)
        r.sweep(8)
        hist = g.pressure()[2]
        assert np.array_equal(hist, r.histogram(200, 1e-4))
        seen += int(hist.sum())
    assert seen > 0

