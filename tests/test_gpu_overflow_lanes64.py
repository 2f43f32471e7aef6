"""FP64 passes with several lanes per particle where every list overflows
(smoothing lengths of 2.6 to 3 dp in 2-D, 1.8 dp in 3-D, more neighbours than
the lists' 96 and 128 entries) or some do: one step and its adjoint against the
oracle, at 16, 8, 4 and 1 lanes per particle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2411_13992_gb300 as sph
from paper_2411_13992_gb300 import cases

from gpu_helpers import compare_step, normwise, oracle_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    assert torch.cuda.is_available()
    oracle.set_threads(16)


def _wide(c, f):
    c = dict(c)
    c["h"] = c["h"] * f
    c["h_min"], c["h_max"] = f * c["h_min"], f * c["h_max"]
    return c


def _varying(c):
    """Half of the particles with more neighbours than a list holds."""
    c = dict(c)
    c["h"] = c["h"] * np.where(np.arange(c["n"]) % 2, 2.4, 1.2)
    c["h_min"], c["h_max"] = float(c["h"].min()), float(c["h"].max())
    return c


CASES = {
    "2d 24": lambda: _wide(cases.tgv2d(24, jitter_dp=0.15), 2.3),
    "2d 70": lambda: _wide(cases.tgv2d(70, jitter_dp=0.15), 2.05),
    "2d 110": lambda: _wide(cases.tgv2d(110, jitter_dp=0.15), 2.3),
    "2d 200": lambda: _wide(cases.tgv2d(200, jitter_dp=0.15), 2.3),
    "2d walls": lambda: _wide(cases.cavity2d(30, jitter_dp=0.15), 2.3),
    "2d varying": lambda: _varying(cases.tgv2d(40, jitter_dp=0.15)),
    "3d 12": lambda: _wide(cases.tgv3d(12, jitter_dp=0.15), 1.4),
    "3d 17": lambda: _wide(cases.tgv3d(17, jitter_dp=0.15), 1.4),
    "3d 24": lambda: _wide(cases.tgv3d(24, jitter_dp=0.15), 1.4),
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_step(case):
    c = CASES[case]()
    P = oracle_params(c)
    s0 = oracle.sigma0_for(c, c["dim"])
    fp = oracle.force_pass(P, c, c["x"], c["v"], s0)
    state = {"x": c["x"], "v": c["v"], "a": fp["a"], "dr": fp["dr"]}
    err, _, _ = compare_step(c, state, oracle.time_step(P, c["v"], c["kind"]), s0, P, precision=64)
    for k in ("x", "v", "rho"):
        assert err[k] <= 1e-12, err
    assert err["a"] <= max(1e-12, 4.0 * err["floor_a"]), err


@pytest.mark.parametrize("case", ["2d 24", "2d 110", "2d walls", "2d varying", "3d 12"])
def test_reverse_step(case):
    """Within the FP64 bound of the adjoint tests; d/d(eta), a sum over all pairs,
    within 1e-12 of the sum of its terms' sizes (at most some 1e2 |er| here)."""
    c = CASES[case]()
    n, dim = c["n"], c["dim"]
    P = oracle_params(c)
    s0 = oracle.sigma0_for(c, dim)
    dt = 0.5 * oracle.time_step(P, c["v"], c["kind"])
    rng = np.random.default_rng(n)
    wts = {k: np.zeros((n, 3)) for k in ("x", "v", "a", "dr")}
    for k, scale in (("x", 1.0), ("v", 1.0), ("a", 1e-2), ("dr", 1e3)):
        wts[k][:, :dim] = rng.standard_normal((n, dim)) * scale
    states = oracle.rollout(P, c, c["x"], c["v"], s0, dt, 1)
    xr, vr, er = oracle.rollout_adjoint(P, c, states, s0, dt, wts)
    sim = sph.Simulation(c, precision=64, fixed_dt=dt, adjoint_steps=1)
    try:
        sim.set_state()
        sim.build_cells()
        st = sim.get_state()
        xb, vb, ab, drb = (wts[k].copy() for k in ("x", "v", "a", "dr"))
        eb = sph.sph_step_adjoint(sim.ctx, st["x"], st["v"], st["a"], st["dr"], 1, xb, vb, ab, drb)
        eb += sph.sph_force_pass_adjoint(sim.ctx, c["x"], c["v"], ab, drb, xb, vb)
        sim.sync()
    finally:
        sim.close()
    fl = c["kind"] == 0
    assert normwise(xb[fl], xr[fl]) <= 1e-12 and normwise(vb[fl], vr[fl]) <= 1e-12
    assert abs(eb - er) <= 1e-10 * max(abs(er), 1.0), (eb, er)
