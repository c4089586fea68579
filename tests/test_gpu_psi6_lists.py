"""psi_6 of every disk against the oracle where the kernel's neighbour lists
can go wrong: cutoffs that reach the corner cells, crowded cells and long
cutoffs (a lane's list is evaluated before the scan ends, a warp's lists
exceed one part of terms), grids of four cells and ragged rows.  psi_6 of a
disk is the same number in every binary64 bit."""
import numpy as np
import pytest

import oracle as O
from paper_1211_1646_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PREC = {"fp64": O.FP64, "fp32": O.FP32}


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("nx,ny,phi,cells,rcut", [
    (4, 4, 0.60, "sigma", 1.4),         # a grid of four cells per axis: images on both sides are one cell
    (70, 62, 0.70, "sigma", 1.4),       # ragged half grid, corner cells out of reach
    (70, 62, 0.70, "sigma", 1.45),      # corner cells within reach
    (33, 38, 0.72, "sigma", 2.0),       # two rings of cells
    (150, 98, 0.708, "sqrt2", 1.4),     # crowded cells
    (90, 62, 0.716, "sqrt2", 2.7),      # crowded cells, about 26 neighbours a disk
    (40, 30, 0.70, "sigma", 1e-3),      # no neighbours
])
def test_psi6_of_every_disk(prec, nx, ny, phi, cells, rcut):
    from paper_1211_1646_gb300 import build, hdmc
    build.build()
    Lx, Ly = W.hex_box(nx, ny, phi)
    g = hdmc.System(nx * ny, Lx, Ly, 1.0, 0.08, 4, 5, prec, cells=cells)
    o = O.System(nx * ny, Lx, Ly, 1.0, 0.08, 4, 5, PREC[prec], cells=O.CELLS_SQRT2 if cells == "sqrt2" else O.CELLS_SIGMA)
    g.sweep(12)
    o.sweep(12)
    mean, mabs, mnb, psi = g.psi6(rcut, per_disk=True)
    ref, ref_psi = o.psi6(rcut, per_disk=True)
    assert np.array_equal(psi, ref_psi)
    N = nx * ny
    assert mnb == ref[3] / N
    assert abs(mean - complex(ref[0], ref[1]) / N) < 1e-12 and abs(mabs - ref[2] / N) < 1e-12
