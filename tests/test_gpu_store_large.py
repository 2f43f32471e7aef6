"""The read-back of a large state into device memory, whose outputs go in one
kernel or one by one through the inverse permutation (the line is at 40 MiB of
output): every choice of outputs, in an order of particles that is not
the order of space, gives the caller's values bit for bit as host memory gets
them."""
import numpy as np
import pytest
import torch

import paper_2411_13992_gb300 as sph
from paper_2411_13992_gb300 import cases

pytestmark = pytest.mark.gpu

CHOICES = [(0, 1, 2, 3, 4), (0,), (4,), (0, 1), (1, 3, 4), (2, 4)]


# 403,298 particles fill 40 MiB with all outputs, 1,747,626 with one vector
@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("n", [403298, 403299, 1747626, 1747627])
def test_large_states_out(precision, n):
    side = int(np.ceil(np.sqrt(n)))
    c = dict(cases.tgv2d(side))
    perm = np.random.default_rng(n).permutation(side * side)[:n]
    for k in ("x", "v", "h", "m", "kind", "vw"):
        c[k] = np.ascontiguousarray(c[k][perm])
    c["n"] = n
    sim = sph.Simulation(c, precision=precision)
    try:
        sim.set_state()
        sim.build_cells()
        sim.sync()
        want = sim.get_state()
        assert np.array_equal(want["x"], c["x"]) and np.abs(want["rho"]).min() > 0.0
        want = [want[k] for k in ("x", "v", "a", "dr", "rho")]
        for choice in CHOICES:
            out = [None] * 5
            for k in choice:
                out[k] = torch.full((n,) if k == 4 else (n, 3), 7.0, dtype=torch.float64, device="cuda")
            sph.sph_get_state(sim.ctx, *out)
            for k in choice:
                assert np.array_equal(out[k].cpu().numpy(), want[k]), (choice, k)
        sim.sync()
    finally:
        sim.close()
