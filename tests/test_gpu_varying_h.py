"""The FP32 step at variable resolution on both sides of the line between a
small grid and one of several waves (512 particles per SM), in 2-D with walls
and in 3-D: one step against the oracle within the FP32 bounds of the parity
tests."""
import numpy as np
import pytest
import torch

import oracle
from paper_2411_13992_gb300 import cases

from gpu_helpers import compare_step, oracle_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    assert torch.cuda.is_available()
    oracle.set_threads(16)


def _varying_3d(side):
    c = dict(cases.tgv3d(side, jitter_dp=0.1))
    c["h"] = c["h"] * (1.0 + 0.15 * np.sin(c["x"][:, 0]) ** 2)
    c["h_min"], c["h_max"] = float(c["h"].min()), float(c["h"].max())
    return c


@pytest.mark.parametrize("case,small", [(lambda: cases.cylinder2d(res=3, jitter_dp=0.05), True),
                                        (lambda: cases.cylinder2d(res=10, jitter_dp=0.05), True),
                                        (lambda: cases.cylinder2d(res=11, jitter_dp=0.05), False),
                                        (lambda: _varying_3d(12), True), (lambda: _varying_3d(44), False)])
def test_step_on_both_sides_of_the_line(case, small):
    c = case()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert (c["n"] <= 512 * sms) == small
    P = oracle_params(c)
    s0 = oracle.sigma0_for(c, c["dim"])
    fp = oracle.force_pass(P, c, c["x"], c["v"], s0)
    state = {"x": c["x"], "v": c["v"], "a": fp["a"], "dr": fp["dr"]}
    err, _, _ = compare_step(c, state, oracle.time_step(P, c["v"], c["kind"]), s0, P, precision=32)
    for k in ("x", "v", "rho"):
        assert err[k] <= 1e-5, err
    assert err["a"] <= max(1e-3, 4.0 * err["floor_a"]), err
