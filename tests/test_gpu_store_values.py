"""The read-back of single outputs of an FP32 state in device memory gives the
stored values exactly (zeros of both signs, subnormal and the largest numbers
among them), and the bits that the read-back of all outputs gives."""
import numpy as np
import pytest
import torch

import paper_2411_13992_gb300 as sph
from paper_2411_13992_gb300 import cases

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,side", [(2, 9), (3, 9), (2, 141), (2, 142), (3, 28)])     # the conversion changes at 20,000
def test_single_outputs_of_extreme_values(dim, side):
    c = (cases.tgv2d if dim == 2 else cases.tgv3d)(side, jitter_dp=0.1)
    n = c["n"]
    rng = np.random.default_rng(1)
    special = np.array([0.0, -0.0, 1e-45, -1e-45, 1.1754942e-38, -1.17549435e-38, 3.4028235e38, -3.4028235e38, 1.0])
    v, a, dr = (np.float32(np.where(rng.random((n, 3)) < 0.5, rng.choice(special, (n, 3)), rng.standard_normal((n, 3))))
                .astype(np.float64) for _ in range(3))
    for q in (v, a, dr):
        q[:, dim:] = 0.0
    sim = sph.Simulation(c, precision=32)
    try:
        sph.sph_set_state(sim.ctx, c["x"], v, a, dr, c["h"], c["m"], c["kind"], c["vw"])
        want = (c["x"], v, a, dr)
        for k in range(4):
            out = [None] * 4
            out[k] = torch.full((n, 3), 7.0, dtype=torch.float64, device="cuda")
            sph.sph_get_state(sim.ctx, *out)
            got = out[k].cpu().numpy()
            assert np.array_equal(got, want[k]) and np.array_equal(np.signbit(got), np.signbit(want[k]))
        sph.sph_set_state(sim.ctx, c["x"], c["v"], None, None, c["h"], c["m"], c["kind"], c["vw"])
        sim.build_cells()
        alone = torch.zeros(n, dtype=torch.float64, device="cuda")
        sph.sph_get_state(sim.ctx, None, None, None, None, alone)
        assert np.array_equal(alone.cpu().numpy(), sim.get_state()["rho"])
        sim.sync()
    finally:
        sim.close()
