"""The votes and sums of the sub-sweeps need every lane of a warp.  A build with
-DHDMC_CHECK_WARPS tests in front of each that a vote reaches the whole warp and
reports HDMC_ECHECK where it does not; the kernels are otherwise the product's.
Run in a separate process on systems with enough pairs near contact that lanes of
one warp decide trials in binary64 together, some to accept and some to reject."""
import os
import subprocess
import sys
import textwrap

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = textwrap.dedent('''
    import os
    import sys
    sys.path.insert(0, %r)
    from paper_1211_1646_gb300 import build, hdmc, workloads as W

    build.OUT_DIR = sys.argv[1]
    build.LIB = os.path.join(build.OUT_DIR, "libhdmc.so")
    lib = build.build(force=True, extra=("-DHDMC_CHECK_WARPS",))
    hdmc.library_path = lambda: lib

    failed = []

    def run(what, s, sweeps):
        try:
            s.sweep(sweeps)
            if hasattr(s, "autotune"):
                s.autotune(4)
            s.counters()
            if hasattr(s, "sync"):
                s.sync()
            else:
                s.pressure()
        except hdmc.HDMCError as e:
            failed.append((what, e.code))

    for prec in ("fp64", "fp32"):
        for nx, ny, phi, cells, nsel, sweeps in [
            (32, 32, 0.70, "sigma", 4, 4000),         # binary64: 8 lanes per cell
            (61, 62, 0.72, "sqrt2", 7, 1000),         # crowded cells
            (233, 254, 0.70, "sigma", 4, 300),        # 4 lanes
            (331, 350, 0.70, "sigma", 5, 200),        # 2 lanes
            (1024, 1024, 0.716, "sigma", 4, 60),      # one thread, n_M fixed
            (1024, 1024, 0.70, "sigma", 8, 60),
            (800, 810, 0.66, "sigma", 11, 40),        # one thread, run-time n_M
        ]:
            Lx, Ly = W.hex_box(nx, ny, phi)
            run((prec, nx, nsel, cells), hdmc.System(nx * ny, Lx, Ly, 1.0, 0.11, nsel, 23, prec, cells=cells), sweeps)
        for q, nsel, sweeps in [(8, 4, 2000), (22, 4, 200), (40, 8, 40)]:
            w = W.fcc3(q, 0.47, 0.1)
            run((prec, "spheres", q, nsel), hdmc.System3(w.N, w.L, 1.0, w.d, nsel, 11, prec), sweeps)
        run((prec, "batch"), hdmc.Batch(W.batch64(seed=3, R=8, nmin=4096, nmax=65536), precision=prec), 64)
    print("failed", failed)
    assert not failed, failed
''') % ROOT


def test_votes_reach_the_whole_warp(tmp_path):
    r = subprocess.run([sys.executable, "-c", SCRIPT, str(tmp_path)], capture_output=True, text=True, timeout=1200)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
