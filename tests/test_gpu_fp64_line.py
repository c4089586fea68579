"""Binary64 systems on either side of the number of active cells from which one
thread updates a cell, with shifts that read the own cell early and late, against
the oracle, bit for bit."""
import numpy as np
import pytest

import oracle as O
from paper_1211_1646_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nsel", [
    (331, 350, 8),     # 32,336 active cells: two lanes
    (340, 350, 4),     # 33,200: one thread, shifts read early
    (340, 350, 8),
    (340, 350, 11),
    (440, 430, 4),     # above 200,000 cells: shifts read late
])
def test_either_side_of_the_line(nx, ny, nsel):
    from paper_1211_1646_gb300 import build, hdmc
    build.build()
    Lx, Ly = W.hex_box(nx, ny, 0.70)
    g = hdmc.System(nx * ny, Lx, Ly, 1.0, 0.11, nsel, 23, "fp64")
    r = O.System(nx * ny, Lx, Ly, 1.0, 0.11, nsel, 23, O.FP64)
    assert (g.C // 4 > 32768) == (nx != 331) and (g.C > 200000) == (nx == 440)
    g.sweep(6)
    r.sweep(6)
    lg, cg = g.state()
    lr, cr = r.state()
    assert np.array_equal(cg, cr)
    assert np.array_equal(lg, lr)
    assert np.array_equal(g.counters(), r.counters())
    assert np.array_equal(g.origin(), r.origin())
