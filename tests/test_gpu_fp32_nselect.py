"""The binary32 sub-sweep at every n_M that is fixed at compile time, in warps
whose cells hold at most two disks and in warps with fuller cells, against the
oracle, bit for bit."""
import numpy as np
import pytest

import oracle as O
from paper_1211_1646_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nsel", [1, 2, 3, 4, 5, 6, 7, 8, 9])
@pytest.mark.parametrize("nx,ny,phi", [(75, 70, 0.70),   # cells of about sigma
                                       (5, 62, 0.723)])  # columns of wide cells (1.4 sigma): up to four disks
def test_every_fixed_nselect(nx, ny, phi, nsel):
    from paper_1211_1646_gb300 import build, hdmc
    build.build()
    Lx, Ly = W.hex_box(nx, ny, phi)
    g = hdmc.System(nx * ny, Lx, Ly, 1.0, 0.13, nsel, 41, "fp32")
    r = O.System(nx * ny, Lx, Ly, 1.0, 0.13, nsel, 41, O.FP32)
    for shuffle in (True, False):
        g.set_balance(shuffle, True)
        r.set_balance(shuffle, True)
        g.sweep(15)
        r.sweep(15)
        lg, cg = g.state()
        lr, cr = r.state()
        assert np.array_equal(cg, cr)
        assert np.array_equal(lg, lr)
        assert np.array_equal(g.counters(), r.counters())
