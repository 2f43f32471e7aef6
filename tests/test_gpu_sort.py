"""The counting sort at the sizes where its kernels change form: fewer bins
than particles and more, one scan tile of 8,192 bins and several, a last tile
that is not full, bins that hold many particles.  The sort's order is fixed by
the bins and the ids alone, so a state loaded in another order gives the same
sums, particle by particle, as the FP64 density of the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2411_13992_gb300 as sph
from paper_2411_13992_gb300 import cases

from gpu_helpers import oracle_params

pytestmark = pytest.mark.gpu


def _density(c, precision, order=None, **kw):
    c = dict(c)
    if order is not None:
        for k in ("x", "v", "h", "m", "kind", "vw"):
            c[k] = np.ascontiguousarray(c[k][order])
    sim = sph.Simulation(c, precision=precision, **kw)
    try:
        sim.set_state()
        sim.build_cells()
        sim.sync()
        rho = sim.get_state()["rho"]
    finally:
        sim.close()
    if order is not None:
        back = np.empty_like(rho)
        back[order] = rho
        rho = back
    return rho


# bins: 4 x floor(side / 1.3)^2 sub-cells; 8,192 bins lie between sides 58 and 59
@pytest.mark.parametrize("side,x_subcells", [(8, 1), (8, 4), (45, 4), (58, 4), (59, 4), (60, 2), (131, 4), (240, 4)])
def test_density_against_the_oracle(side, x_subcells):
    """FP64 sums of about 21 terms: within 1e-12 (the library's stated FP64 bound)."""
    c = cases.tgv2d(side, jitter_dp=0.2, seed=side)
    P = oracle_params(c)
    ref = oracle.force_pass(P, c, c["x"], c["v"], oracle.sigma0_for(c, 2))["rho"]
    got = _density(c, 64, x_subcells=x_subcells)
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("precision", [64, 32])
def test_loading_order_changes_the_sums_by_rounding_only(precision):
    """A shuffled load gives other ids and so another order within the bins:
    sums of the same terms, within 21 roundings of the term size."""
    c = cases.tgv2d(59, jitter_dp=0.2, seed=5)
    rng = np.random.default_rng(1)
    a = _density(c, precision)
    b = _density(c, precision, order=rng.permutation(c["n"]))
    eps = np.finfo(np.float64 if precision == 64 else np.float32).eps
    assert np.abs(a - b).max() <= 21 * 4 * eps * np.abs(a).max()


def test_bins_of_many_particles():
    """2,000 particles in a few bins of a 2-D box (beyond the list's capacity,
    so the force pass scans the cells): the order by id within a bin is found
    for every one of them, and two loads agree bit for bit."""
    c = dict(cases.tgv2d(50))
    rng = np.random.default_rng(2)
    x = c["x"].copy()
    crowd = rng.choice(c["n"], 2000, replace=False)
    x[crowd, :2] = 0.5 + 0.01 * (rng.random((2000, 2)) - 0.5)
    c["x"] = x
    a = _density(c, 64)
    b = _density(c, 64)
    assert np.array_equal(a, b)
    P = oracle_params(c)
    ref = oracle.force_pass(P, c, x, c["v"], oracle.sigma0_for(c, 2))["rho"]
    assert np.abs(a - ref).max() <= 1e-12 * np.abs(ref).max()
