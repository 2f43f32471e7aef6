"""Pairs so close that r^2 is a subnormal number in the pass's precision
(1e-20 in FP32, 1e-160 in FP64): distinct particles, so the pair's viscous term
counts (W'(r)/r stays finite) and the others vanish with r.  Density,
acceleration and displacement stay finite and on the oracle's."""
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


def _close_pair(c, gap):
    """Particle 0 moved to the corner of the box (offset 0 from its cell's
    origin, where a gap this small is still a gap), and a twin beside it."""
    for k in ("x", "v", "h", "m", "kind", "vw"):
        c[k] = np.ascontiguousarray(np.concatenate([c[k], c[k][:1]]))
    c["n"] += 1
    assert tuple(c["lo"]) == (0.0, 0.0, 0.0)
    c["x"][0] = 0.0
    c["x"][-1] = (gap, 0.0, 0.0)
    c["v"][0, 0], c["v"][-1, 0] = 0.3, -0.2
    return c


# the bounds of the parity tests: FP64 1e-12; FP32 1e-5 (rho) and 1e-3 (a, dr)
@pytest.mark.parametrize("precision,gap,tol_rho,tol_a", [(64, 1e-160, 1e-12, 1e-12), (64, 1e-20, 1e-12, 1e-12),
                                                         (32, 1e-20, 1e-5, 1e-3), (32, 3e-22, 1e-5, 1e-3)])
@pytest.mark.parametrize("dim", [2, 3])
def test_force_pass_of_a_close_pair(dim, precision, gap, tol_rho, tol_a):
    c = _close_pair((cases.tgv2d if dim == 2 else cases.tgv3d)(16, jitter_dp=0.1, seed=5), gap)
    ref = oracle.force_pass(oracle_params(c), c, c["x"], c["v"], oracle.sigma0_for(c, dim))
    sim = sph.Simulation(c, precision=precision)
    try:
        sim.set_state()
        sim.build_cells()
        got = sim.get_state()
        assert sim.sync() is None
    finally:
        sim.close()
    assert normwise(got["rho"], ref["rho"]) <= tol_rho
    for k in ("a", "dr"):
        assert np.isfinite(got[k]).all(), k
        assert normwise(got[k], ref[k]) <= tol_a, k
