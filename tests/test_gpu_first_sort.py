"""The first sort of a large loaded state (1.5 million particles or more), which
ranks and moves the particles in two kernels: bit for bit what the sort of one
kernel makes of the same particles, whatever order they are loaded in."""
import numpy as np
import pytest
import torch

import paper_2411_13992_gb300 as sph
from paper_2411_13992_gb300 import cases

pytestmark = pytest.mark.gpu

SIDE = 1225                       # 1,500,625 particles
KEYS = ("x", "v", "a", "dr", "rho")


def _case(share, n=SIDE * SIDE):
    """The vortex with a share of its particles loaded in places of others."""
    c = dict(cases.tgv2d(SIDE, jitter_dp=0.1))
    rng = np.random.default_rng(int(100 * share))
    perm = np.arange(SIDE * SIDE)
    pick = rng.choice(len(perm), int(share * len(perm)), replace=False)
    perm[pick] = pick[rng.permutation(len(pick))]
    for k in ("x", "v", "h", "m", "kind", "vw"):
        c[k] = np.ascontiguousarray(c[k][perm[:n]])
    c["n"] = n
    return c


def _same(s, t, keys=KEYS):
    for k in keys:
        assert np.array_equal(s[k], t[k]), k


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("share", [0.0, 0.3, 1.0])
def test_built_again_from_the_sorted_state(precision, share):
    sim = sph.Simulation(_case(share), precision=precision)
    try:
        sim.set_state()
        sim.build_cells()
        first = sim.get_state()
        sim.build_cells()                  # sorts the sorted particles, in one kernel
        _same(first, sim.get_state())
        assert sim.sync() is None
    finally:
        sim.close()


@pytest.mark.parametrize("share,n", [(1.0, SIDE * SIDE), (1.0, 1500000), (1.0, 1499999), (0.0, 1500000)])
def test_varying_constants_and_given_accelerations(share, n):
    """h, masses and walls that travel with the sort; a and dr given: a read of
    the density sorts the loaded state, or the first step does."""
    c = _case(share, n)
    rng = np.random.default_rng(4)
    c["m"] = c["m"] * (1.0 + 0.01 * rng.random(n))
    c["h"] = c["h"] * (1.0 + 0.1 * rng.random(n))
    c["h_min"], c["h_max"] = float(c["h"].min()), float(c["h"].max())
    c["kind"] = (rng.random(n) < 0.02).astype(np.int8)
    ad = [1e-3 * rng.standard_normal((n, 3)), 1e-3 * c["dp"] * rng.standard_normal((n, 3))]
    for q in ad:
        q[:, 2] = 0.0
        q[c["kind"] != 0] = 0.0
    runs = []
    for read_first in (True, False):
        sim = sph.Simulation(c, precision=32)
        try:
            sim.set_state(a=ad[0], dr=ad[1])
            sim.build_cells()
            if read_first:
                s = sim.get_state()
                assert np.array_equal(s["x"], c["x"]) and np.array_equal(s["a"], ad[0].astype(np.float32))
            sim.step(3)
            runs.append(sim.get_state())
            assert sim.sync() is None
        finally:
            sim.close()
    _same(*runs)


@pytest.mark.parametrize("share", [0.0, 1.0])
def test_adjoint_segment_recorded_and_launched(share):
    c = _case(share)
    n = c["n"]
    out = []
    for graphs in (1, 0):
        rng = np.random.default_rng(6)
        sim = sph.Simulation(c, precision=32, graphs=graphs, fixed_dt=1e-3 * c["dp"], adjoint_steps=1)
        try:
            sim.set_state()
            sim.build_cells()
            s = sim.get_state()
            for _ in range(2):
                bars = [rng.standard_normal((n, 3)) for _ in range(4)]
                for b in bars:
                    b[:, 2] = 0.0
                eta = sph.sph_step_adjoint(sim.ctx, s["x"], s["v"], s["a"], s["dr"], 1, *bars)
                out.append((graphs, bars, eta, sim.get_state()))
            assert sim.sync() is None
        finally:
            sim.close()
    for (_, b1, e1, s1), (_, b0, e0, s0) in zip(out[:2], out[2:]):
        assert e1 == e0 and all(np.array_equal(p, q) for p, q in zip(b1, b0))
        _same(s1, s0)


@pytest.mark.parametrize("precision", [32, 64])
def test_dual_integrator_carries_the_density_rate(precision):
    c = _case(1.0)
    rate = np.random.default_rng(9).standard_normal(c["n"])
    if precision == 32:
        rate = rate.astype(np.float32).astype(np.float64)
    sim = sph.Simulation(c, precision=precision, integrator=sph.INT_DUAL)
    try:
        sim.set_state(drho=rate)
        sim.build_cells()
        first = sim.get_state()
        assert np.array_equal(sim.density_rate(), rate)
        sim.build_cells()
        _same(first, sim.get_state(), ("x", "v", "rho"))     # (a and dr are the first step's)
        assert np.array_equal(sim.density_rate(), rate)
        sim.sync()
    finally:
        sim.close()
