"""The work that a user of this library has it do, as cases to be timed.

A pass is what a simulation program repeats: a run of Monte Carlo sweeps, the
contact histogram and pressure of the configuration it ends in, and the
configuration itself (a checkpoint image in pinned host memory for the large
systems, the raw state or the global coordinates for the others); or the
analysis of a configuration alone.  Sizes, densities, move sizes and sweep
counts are those of paper_1211_1646_gb300/workloads.py, bench.py and the
tests.  The systems start from the library's lattice and are run for a while
before they are measured, so that the cells hold a fluid, not a lattice.

Kinds of case
  disks    one hard-disk system (hdmc.System): sweeps, pressure, state
  batch    replicas advanced together (hdmc.Batch)
  spheres  one hard-sphere system (hdmc.System3)
  observe  contact histogram, pressure and psi_6 of a disk configuration
"""
import math

import numpy as np
import torch

from paper_1211_1646_gb300 import hdmc, workloads

R_CUT = 1.4   # psi_6 neighbour distance (the library's default)


def _disks(name, nx, ny, phi, d, nselect, precision, sweeps, out, cells="sigma", box="hex"):
    return {"name": name, "kind": "disks", "nx": nx, "ny": ny, "phi": phi, "box": box, "d": d, "nselect": nselect,
            "precision": precision, "cells": cells, "sweeps": sweeps, "out": out}


def listed():
    return [
        # the smallest workload: 1024 disks in binary64, its 200 sweeps (launch latency; tests and checks of a set-up)
        _disks("disks_n1024_f64", 32, 32, 0.70, 0.15, 4, "fp64", 200, "state", box="square"),
        # 256^2 disks in binary64, one pressure every 100 sweeps: a Table 1 sized equation-of-state run
        _disks("disks_n65536_f64", 256, 256, 0.70, 0.10, 4, "fp64", 100, "save", box="square"),
        # a system of the replicas' lower sizes with a grid of odd half-width and n_M = 7: the run-time n_M
        _disks("disks_ragged_f32_nm7", 94, 110, 0.68, 0.12, 7, "fp32", 100, "state"),
        # the headline workload: 1024^2 disks, binary32, 100 sweeps + histogram + fit
        _disks("disks_n1m_f32", 1024, 1024, 0.716, 0.08, 4, "fp32", 100, "save"),
        # the same in binary64
        _disks("disks_n1m_f64", 1024, 1024, 0.716, 0.08, 4, "fp64", 100, "save"),
        # 2048^2 disks: a state larger than the L2 cache
        _disks("disks_n4m_f32", 2048, 2048, 0.710, 0.08, 4, "fp32", 100, "save"),
        # the paper's Table 4 workload: 1520^2 disks in cells just below sqrt(2) sigma
        _disks("disks_table4_f32", 1520, 1520, 0.698, 0.16, 4, "fp32", 100, "save", cells="sqrt2", box="square"),
        # 64 replicas of 4096 to 262144 disks at n_M = 8 (what the batch's tuner picks for them)
        {"name": "batch64_f32_nm8", "kind": "batch", "R": 64, "nmin": 4096, "nmax": 262144, "shape": 1, "nselect": 8,
         "precision": "fp32", "sweeps": 100},
        # the smallest sphere workload, binary64
        {"name": "spheres_n2048_f64", "kind": "spheres", "q": 8, "phi": 0.45, "d": 0.10, "nselect": 4,
         "precision": "fp64", "sweeps": 100},
        # the middle sphere workload, binary32
        {"name": "spheres_n16384_f32", "kind": "spheres", "q": 16, "phi": 0.45, "d": 0.10, "nselect": 4,
         "precision": "fp32", "sweeps": 100},
        # a million spheres at the freezing density: sweeps, pressure and one trajectory frame
        {"name": "spheres_n1m_f32", "kind": "spheres", "q": 64, "phi": 0.49, "d": 0.08, "nselect": 4,
         "precision": "fp32", "sweeps": 400},
        # the analysis of one configuration of the headline workload (Sec. 4's histogram, Sec. 3.3's order parameter)
        {"name": "observe_n1m_f32", "kind": "observe", "nx": 1024, "ny": 1024, "phi": 0.716, "box": "hex",
         "precision": "fp32", "cells": "sigma", "per_disk": False},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _spheres_fit(q, phi):
    """Whether the fcc workload of q^3 unit cells has a legal cell grid (w_x^2 + w_y^2 + w_z^2 < 4 sigma^2)."""
    L = workloads.cube_box3(4 * q ** 3, phi)[0]
    m = 2 * (int(L) // 2)
    return m >= 4 and 3.0 * (L / m) ** 2 < 3.99


def draw(rng):
    kind = rng.choices(["disks", "batch", "spheres", "observe"], [5, 1, 3, 1])[0]
    precision = rng.choice(["fp32", "fp64"])
    nselect = rng.choices([4, 8, rng.randint(1, 12)], [5, 2, 3])[0]
    if kind in ("disks", "observe"):
        most = 1048576 if precision == "fp64" or kind == "observe" or nselect > 8 else 4194304
        nx, ny = workloads.hex_counts(int(_log_uniform(rng, 1024, most)))
        c = {"kind": kind, "nx": nx, "ny": ny, "phi": round(rng.uniform(0.60, 0.72), 4), "box": "hex",
             "precision": precision, "cells": rng.choice(["sigma", "sigma", "sqrt2"])}
        if kind == "disks":
            c.update(d=round(rng.uniform(0.05, 0.16), 4), nselect=nselect, sweeps=rng.randint(50, 100),
                     out="state" if nx * ny < 20000 else "save")
        else:   # psi_6 of every disk (a map of the order parameter), or the means alone
            c.update(per_disk=nx * ny < 100000)
        return c
    if kind == "batch":
        R = int(_log_uniform(rng, 4, 64))
        return {"kind": "batch", "R": R, "nmin": 1024, "nmax": rng.choice([8192, 32768, 131072]),
                "shape": rng.randint(2, 10 ** 6), "nselect": min(nselect, 8), "precision": precision,
                "sweeps": 100 if precision == "fp32" else 40}
    while True:
        q, phi = int(_log_uniform(rng, 8, 64 if precision == "fp32" else 40)), round(rng.uniform(0.40, 0.49), 4)
        if _spheres_fit(q, phi):
            return {"kind": "spheres", "q": q, "phi": phi, "d": round(rng.uniform(0.05, 0.12), 4),
                    "nselect": min(nselect, 8), "precision": precision, "sweeps": rng.randint(50, 100)}


def _box(case):
    if case["box"] == "square":
        return workloads.square_box(case["nx"] * case["ny"], case["phi"])
    return workloads.hex_box(case["nx"], case["ny"], case["phi"])


def _replicas(case):
    """The batch's systems: sizes and densities from the case alone."""
    return workloads.batch64(seed=case["shape"], R=case["R"], nmin=case["nmin"], nmax=case["nmax"])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        reps = _replicas(case)
        for r, w in enumerate(reps):
            w.nselect, w.seed = case["nselect"], seed * 1000003 + r
        b = hdmc.Batch(reps, precision=case["precision"])
        b.sweep(200 if case["precision"] == "fp32" else 50)
        return {"kind": kind, "sys": b, "sweeps": case["sweeps"],
                "buf": torch.empty(b.snapshot_bytes(), dtype=torch.uint8, pin_memory=True)}
    if kind == "spheres":
        w = workloads.fcc3(case["q"], case["phi"], case["d"], nselect=case["nselect"])
        s = hdmc.System3(w.N, w.L, 1.0, w.d, w.nselect, seed, case["precision"])
        s.sweep(100 if w.N < 500000 else 40)
        return {"kind": kind, "sys": s, "sweeps": case["sweeps"], "frame": w.N > 500000}
    N = case["nx"] * case["ny"]
    Lx, Ly = _box(case)
    s = hdmc.System(N, Lx, Ly, 1.0, case.get("d", 0.08), case.get("nselect", 4), seed, case["precision"],
                    cells=case["cells"])
    s.sweep(1000 if N < 100000 and case["precision"] == "fp32" else 200)
    state = {"kind": kind, "sys": s, "per_disk": case.get("per_disk", False)}
    if kind == "disks":
        state["sweeps"] = case["sweeps"]
        if case["out"] == "save":
            state["buf"] = torch.empty(s.snapshot_bytes(), dtype=torch.uint8, pin_memory=True)
    return state


def run(state):
    s = state["sys"]
    if state["kind"] == "observe":
        s.sample()
        bp, g0, hist, ns = s.pressure()
        mean, mabs, mnb, *psi = s.psi6(R_CUT, per_disk=state["per_disk"])
        return {"betaP_over_rho": bp, "g_contact": g0, "hist": hist,
                "psi6": [mean.real, mean.imag, float(mabs), float(mnb)], "psi6_of_disks": psi}
    s.sweep(state["sweeps"])
    s.sample()
    bp, g0, hist, ns = s.pressure()
    out = {"betaP_over_rho": bp, "g_contact": g0, "hist": hist, "counters": s.counters()}
    if "buf" in state:
        out["image"] = s.save(state["buf"])
    elif state.get("frame"):
        out["positions"] = s.positions()
    else:
        out["local"], out["counts"] = s.state()
    return out


def _particles(case):
    """Particles of a case, summed over a batch's replicas."""
    if case["kind"] == "spheres":
        return 4 * case["q"] ** 3
    if case["kind"] == "batch":
        return sum(w.N for w in _replicas(case))
    return case["nx"] * case["ny"]


def work(case):
    """Bytes: the coordinates read once and written once (8 or 16 bytes a
    disk, 12 or 24 a sphere).  Operations: per trial move, 5 for each other
    particle in reach (7 in three dimensions), 6 for the trial position and
    its containment (9), and the random direction (46 disks, 122 spheres,
    Philox included); each occupied cell makes n_M trial moves a sweep.  Per
    disk of an analysis: 9 for each of the 23 disks of the 5 x 5 cells and 30
    for each of its 6 neighbours."""
    N = _particles(case)
    size = 4 if case["precision"] == "fp32" else 8
    if case["kind"] == "observe":
        return {"bytes": 2.0 * size * N, "flops": N * (9 * 23 + 30 * 6)}
    dense = case.get("cells") == "sqrt2"
    if case["kind"] == "spheres":
        dim, occupied, per_trial = 3, 0.72 * N, 11 * 7 + 9 + 122
    else:
        dim, occupied, per_trial = 2, (0.52 if dense else 0.95) * N, (14 if dense else 7.3) * 5 + 6 + 46
    trials = occupied * case["nselect"] * case["sweeps"]
    return {"bytes": 2.0 * dim * size * N, "flops": trials * per_trial}


def exact(case, seed):
    """The analysis cases in 64 bits: psi_6 and the pressure of the prepared
    configuration.  A trajectory has no such value (its accept decisions make
    it chaotic), so the other cases have none."""
    if case["kind"] != "observe":
        return None
    s = prepare(case, seed)["sys"]
    loc, cnt = s.state()
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    wx, wy = (s.wx, s.wy) if case["precision"] == "fp64" else (float(np.float32(s.wx)), float(np.float32(s.wy)))
    mx, my = s.mx, s.my
    x = torch.from_numpy(loc[:, :, 0].copy()).to(dev).reshape(my, mx, 4)
    y = torch.from_numpy(loc[:, :, 1].copy()).to(dev).reshape(my, mx, 4)
    n = torch.from_numpy(cnt.astype(np.int64)).to(dev).reshape(my, mx, 1)
    has = torch.arange(4, device=dev).reshape(1, 1, 4) < n
    edges = (1.0 + 1.0e-4 * torch.arange(201, dtype=torch.float64, device=dev)) ** 2
    hist = torch.zeros(200, dtype=torch.int64, device=dev)
    re, im = torch.zeros_like(x), torch.zeros_like(x)
    nb = torch.zeros_like(x)
    for dy in range(-2, 3):
        for dx in range(-2, 3):
            for j in range(4):
                qx = torch.roll(x[:, :, j], (-dy, -dx), (0, 1)) + dx * wx
                qy = torch.roll(y[:, :, j], (-dy, -dx), (0, 1)) + dy * wy
                qh = torch.roll(has[:, :, j], (-dy, -dx), (0, 1))
                for i in range(4):
                    if dx == 0 and dy == 0 and i == j:
                        continue
                    pair = has[:, :, i] & qh
                    ex, ey = x[:, :, i] - qx, y[:, :, i] - qy
                    r2 = ex * ex + ey * ey
                    near = r2[pair & (r2 >= edges[0]) & (r2 < edges[200])]
                    if near.numel():
                        b = torch.searchsorted(edges, near, right=True) - 1
                        hist += torch.bincount(b, minlength=200)[:200]
                    bond = pair & (r2 < R_CUT * R_CUT)
                    z = torch.complex(ex, ey)
                    u = torch.where(bond, z / torch.sqrt(torch.where(bond, r2, 1.0)), 0)
                    u6 = (u * u * u) ** 2
                    re[:, :, i] += u6.real
                    im[:, :, i] += u6.imag
                    nb[:, :, i] += bond
    k = torch.clamp(nb, min=1.0)
    N = case["nx"] * case["ny"]
    pr, pi = re / k, im / k
    psi6 = [float(pr.sum()) / N, float(pi.sum()) / N, float(torch.sqrt(pr * pr + pi * pi).sum()) / N,
            float(nb.sum()) / N]
    # g(R_i) and the degree-5 fit over (sigma, 1.02 sigma] at contact (Sec. 4)
    Lx, Ly = _box(case)
    r = 1.0 + 1.0e-4 * np.arange(201)
    R = (2.0 / 3.0) * (r[1:] ** 3 - r[:-1] ** 3) / (r[1:] ** 2 - r[:-1] ** 2)
    rho = N / (Lx * Ly)
    g = hist.cpu().numpy() / (N * rho * 2.0 * np.pi * R * 1.0e-4)
    g0 = float(np.linalg.lstsq(np.vander((R - 1.0) / 0.02, 6, increasing=True), g, rcond=None)[0][0])
    psi = [torch.stack([pr, pi], dim=-1).reshape(mx * my, 4, 2)] if case["per_disk"] else []
    return {"betaP_over_rho": 1.0 + 0.5 * np.pi * rho * g0, "g_contact": g0, "hist": None, "psi6": psi6,
            "psi6_of_disks": psi}
