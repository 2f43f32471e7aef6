"""The FP64 adjoint whose tape is too large to hold its steps' neighbour lists
(more than 1 GiB of them): the reverse sweep builds each step's list again, with
the cotangents of a tape that holds them, bit for bit; the state that the
segment leaves is the same too."""
import numpy as np
import pytest
import torch

import paper_2411_13992_gb300 as sph
from paper_2411_13992_gb300 import cases

pytestmark = pytest.mark.gpu


def _crowded():
    """110 particles within two cells: more neighbours than a list holds."""
    c = dict(cases.tgv2d(40, jitter_dp=0.15, seed=3))
    x = c["x"].copy()
    x[:110, :2] = 0.5 + 2.7 * c["dp"] * np.random.default_rng(5).random((110, 2))
    c["x"] = x
    return c


def _segment(c, adjoint_steps, graphs, nsteps):
    n = c["n"]
    rng = np.random.default_rng(11)
    dt = 0.2 * 0.25 * c["h_min"] / 10.0
    sim = sph.Simulation(c, precision=64, graphs=graphs, fixed_dt=dt, adjoint_steps=adjoint_steps)
    try:
        sim.set_state()
        sim.build_cells()
        s = sim.get_state()
        bars = [rng.standard_normal((n, 3)) for _ in range(4)]
        for b in bars:
            b[:, c["dim"]:] = 0.0
            b[c["kind"] != 0] = 0.0
        eta = sph.sph_step_adjoint(sim.ctx, s["x"], s["v"], s["a"], s["dr"], nsteps, *bars)
        after = sim.get_state()
        eta += sph.sph_force_pass_adjoint(sim.ctx, s["x"], s["v"], bars[2], bars[3], bars[0], bars[1])
        assert sim.sync() is None
        return bars, eta, after, sim.nbytes
    finally:
        sim.close()


@pytest.mark.parametrize("graphs", [1, 0])
@pytest.mark.parametrize("case", [lambda: cases.tgv2d(64, jitter_dp=0.1), lambda: cases.tgv3d(12, jitter_dp=0.1),
                                  lambda: cases.cylinder2d(res=2), _crowded])
def test_rebuilt_lists_give_the_same_bits(case, graphs):
    c = case()
    slot = c["n"] * 4 * ((96 if c["dim"] == 2 else 128) + 1)
    held = (1 << 30) // slot                       # the most slots whose lists the tape holds
    bars, eta, after, nbytes = _segment(c, held, graphs, 4)
    bars2, eta2, after2, nbytes2 = _segment(c, held + 1, graphs, 4)
    assert nbytes2 < nbytes - (1 << 29)
    for a, b in zip(bars, bars2):
        assert np.isfinite(a).all() and np.abs(a).max() > 0.0
        assert np.array_equal(a, b)
    assert eta == eta2
    for k in ("x", "v", "a", "dr", "rho"):
        assert np.array_equal(after[k], after2[k]), k
