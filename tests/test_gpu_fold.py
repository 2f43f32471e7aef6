"""The fold of a pass's partials (diagnostics and the next step size) at the
sizes where it changes form: one block per group or several, a grid that
folds itself or the separate fold kernel, a last block and a last group that
are not full."""
import numpy as np
import pytest
import torch

import paper_2411_13992_gb300 as sph
from paper_2411_13992_gb300 import cases

pytestmark = pytest.mark.gpu

# FP32 blocks hold 128 particles from 152 x 128 on: 256 blocks fold as one
# group, 2,048 in the grid, more in the fold kernel
SIZES = [1, 31, 33, 3000, 256 * 128, 256 * 128 + 1, 2048 * 128, 2048 * 128 + 1, 2049 * 128 + 77]


def _first(n):
    side = max(int(np.ceil(np.sqrt(n))), 8)
    c = dict(cases.tgv2d(side))
    for k in ("x", "v", "h", "m", "kind", "vw"):
        c[k] = np.ascontiguousarray(c[k][:n])
    c["n"] = n
    return c


@pytest.mark.parametrize("given", [False, True])
@pytest.mark.parametrize("n", SIZES)
def test_diagnostics_of_the_loaded_state(n, given):
    """sph_build_cells leaves v as given, so the diagnostics are sums over the
    inputs (velocities rounded to FP32).  A sum of n terms in any order is
    within n eps of the sum of magnitudes; the maxima are exact up to the
    rounding of the FP64 squares."""
    c = _first(n)
    sim = sph.Simulation(c, precision=32)
    try:
        zero = np.zeros((n, 3))
        sim.set_state(a=zero if given else None, dr=zero if given else None)
        sim.build_cells()
        d0 = sim.diag()
        sim.sync()
        again = sim.diag()
    finally:
        sim.close()
    v = c["v"].astype(np.float32).astype(np.float64)
    m = c["m"]
    tol = max(n, 8) * np.finfo(np.float64).eps
    assert abs(d0["mass"] - m.sum()) <= tol * m.sum()
    for k in range(2):
        assert abs(d0["momentum"][k] - (m * v[:, k]).sum()) <= tol * (m * np.abs(v[:, k])).sum()
    ke = 0.5 * (m * (v * v).sum(1)).sum()
    assert abs(d0["ke"] - ke) <= tol * ke
    vmax = np.sqrt((v * v).sum(1)).max()
    assert abs(d0["vmax"] - vmax) <= 4 * np.finfo(np.float64).eps * vmax
    p = sph.params_from_case(c, 32)
    dt = min(p.cfl_ad * p.h_min / max(vmax, p.eta / p.rho0 / p.h_min, p.u_ref), p.cfl_ac * p.h_min / (vmax + p.c0))
    assert abs(d0["dt_next"] - dt) <= 8 * np.finfo(np.float64).eps * dt
    assert {k: np.asarray(x).tolist() for k, x in d0.items()} == {k: np.asarray(x).tolist() for k, x in again.items()}


@pytest.mark.parametrize("n", [3000, 256 * 128 + 1, 2048 * 128 + 1])
def test_the_fold_does_not_depend_on_timing(n):
    """Two runs of the same steps give the same diagnostics bit for bit."""
    c = _first(n)
    out = []
    for _ in range(2):
        sim = sph.Simulation(c, precision=32)
        try:
            sim.set_state()
            sim.build_cells()
            sim.step(3)
            out.append({k: np.asarray(x).tolist() for k, x in sim.diag().items()})
        finally:
            sim.close()
    assert out[0] == out[1]
    assert out[0]["steps"] == 3 and out[0]["n_chi"] <= n
