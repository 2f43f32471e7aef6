"""The FP32 density pass with several lanes per particle, at the sizes where
their number changes (32, 96 and 180 particles per SM) and at the smallest:
bit for bit the states of the walk over shared-memory tiles (pair_tiles = 1
with whole cells, one thread per particle, the same candidates in the same
order), and the densities of lists that overflow against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2411_13992_gb300 as sph
from paper_2411_13992_gb300 import cases

from gpu_helpers import normwise, oracle_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    assert torch.cuda.is_available()


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _first(c, n):
    c = dict(c)
    for k in ("x", "v", "h", "m", "kind", "vw"):
        c[k] = np.ascontiguousarray(c[k][:n])
    c["n"] = n
    return c


def _states(c, **kw):
    sim = sph.Simulation(c, precision=32, x_subcells=1, **kw)
    try:
        sim.set_state()
        sim.build_cells()
        sim.step(3)
        assert sim.sync() is None
        return sim.get_state()
    finally:
        sim.close()


def _same(c, **kw):
    a, b = _states(c, **kw), _states(c, pair_tiles=1, **kw)
    for k in ("x", "v", "a", "dr", "rho"):
        assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("per_sm", [32, 96, 180])
@pytest.mark.parametrize("off", [-1, 0])
def test_both_sides_of_each_line(dim, per_sm, off):
    n = _sms() * per_sm + off
    side = int(np.ceil(n ** (1.0 / dim) - 1e-9))
    _same(_first((cases.tgv2d if dim == 2 else cases.tgv3d)(side, jitter_dp=0.2, seed=n), n))


@pytest.mark.parametrize("compensated", [True, False])
@pytest.mark.parametrize("case", [lambda: cases.cavity2d(37, jitter_dp=0.1), lambda: cases.tgv3d(7),
                                  lambda: _first(cases.tgv2d(20), 1), lambda: _first(cases.tgv3d(9, jitter_dp=0.2), 35)])
def test_walls_wraps_and_few_particles(case, compensated):
    _same(case(), kahan=int(compensated))


@pytest.mark.parametrize("dim", [2, 3])
def test_lists_that_overflow(dim):
    """Most particles in a small part of the box: more neighbours than a list
    holds (96 in 2-D, 128 in 3-D)."""
    c = (cases.tgv2d if dim == 2 else cases.tgv3d)(30 if dim == 2 else 12, jitter_dp=0.2, seed=4)
    c["x"][: c["n"] // 2, :dim] = 0.25 * c["L"][0] + 0.35 * (c["x"][: c["n"] // 2, :dim] - 0.25 * c["L"][0])
    ref = oracle.force_pass(oracle_params(c), c, c["x"], c["v"], oracle.sigma0_for(c, dim))
    sim = sph.Simulation(c, precision=32)
    try:
        sim.set_state()
        sim.build_cells()
        got = sim.get_state()
        assert sim.sync() is None
    finally:
        sim.close()
    assert normwise(got["rho"], ref["rho"]) <= 1e-5
    assert normwise(got["a"], ref["a"]) <= 1e-3
