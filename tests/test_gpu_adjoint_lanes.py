"""The FP64 reverse kernels at the sizes where their lanes per particle change
(128 and 512 particles per SM) and at the smallest: one reverse step against
the oracle's adjoint within the FP64 tolerance of the adjoint tests (1e-12,
normwise).  The list of the forward step is what both forms walk; a particle
with more neighbours than it holds is covered by the adjoint tests."""
import numpy as np
import pytest
import torch

import oracle
import paper_2411_13992_gb300 as sph
from paper_2411_13992_gb300 import cases

from gpu_helpers import normwise, oracle_params

pytestmark = pytest.mark.gpu


def _case(n):
    side = int(np.ceil(np.sqrt(n)))
    c = dict(cases.tgv2d(max(side, 8), jitter_dp=0.12, seed=n))
    for k in ("x", "v", "h", "m", "kind", "vw"):
        c[k] = np.ascontiguousarray(c[k][:n])
    c["n"] = n
    return c


@pytest.mark.parametrize("per_sm,off", [(0, 5), (0, 70), (128, -1), (128, 0), (512, -1), (512, 0)])
def test_fp64_reverse_step(per_sm, off):
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + off
    oracle.set_threads(16)
    c = _case(n)
    P = oracle_params(c)
    s0 = oracle.sigma0_for(c, 2)
    dt = 0.5 * oracle.time_step(P, c["v"], c["kind"])
    rng = np.random.default_rng(n)
    wts = {k: np.zeros((n, 3)) for k in ("x", "v", "a", "dr")}
    for k, scale in (("x", 1.0), ("v", 1.0), ("a", 1e-2), ("dr", 1e3)):
        wts[k][:, :2] = rng.standard_normal((n, 2)) * scale
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
    assert normwise(xb, xr) <= 1e-12 and normwise(vb, vr) <= 1e-12, (normwise(xb, xr), normwise(vb, vr))
    assert abs(eb - er) <= 1e-12 * max(abs(er), 1.0), (eb, er)
