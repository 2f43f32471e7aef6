"""The FP64 pair passes at the sizes where the lanes per particle and the
block size change (the lines lie at 16, 64, 256 and 2,048 particles per SM),
and at the smallest: one step against the oracle within the FP64 tolerances of
the parity tests, and lists that overflow with several lanes per particle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2411_13992_gb300 as sph
from paper_2411_13992_gb300 import cases

from gpu_helpers import compare_step, oracle_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    assert torch.cuda.is_available()
    oracle.set_threads(16)


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _case(dim, n):
    """The first n particles of a jittered periodic vortex."""
    side = int(np.ceil(n ** (1.0 / dim) - 1e-9))
    c = dict((cases.tgv2d if dim == 2 else cases.tgv3d)(max(side, 8), jitter_dp=0.15, seed=n))
    for k in ("x", "v", "h", "m", "kind", "vw"):
        c[k] = np.ascontiguousarray(c[k][:n])
    c["n"] = n
    return c


def _check(c):
    P = oracle_params(c)
    s0 = oracle.sigma0_for(c, c["dim"])
    fp = oracle.force_pass(P, c, c["x"], c["v"], s0)
    state = {"x": c["x"], "v": c["v"], "a": fp["a"], "dr": fp["dr"]}
    err, _, _ = compare_step(c, state, oracle.time_step(P, c["v"], c["kind"]), s0, P, precision=64)
    for k in ("x", "v", "rho"):
        assert err[k] <= 1e-12, err
    assert err["a"] <= max(1e-12, 4.0 * err["floor_a"]), err


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("per_sm", [16, 64, 256])
@pytest.mark.parametrize("off", [-1, 0])
def test_step_on_both_sides_of_each_line(dim, per_sm, off):
    _check(_case(dim, _sms() * per_sm + off))


@pytest.mark.parametrize("n", [1, 2, 37, 511])
def test_step_of_a_few_particles(n):
    _check(_case(2, n))


def test_larger_block_line():
    _check(_case(2, _sms() * 2048))


@pytest.mark.parametrize("n", [600, 12000])
def test_crowded_particles_overflow_the_lists(n):
    """110 particles within two cells have more neighbours than the 96 list
    entries of 2-D: one lane of each group then walks the cells."""
    c = _case(2, n)
    dp = c["dp"]
    x = c["x"].copy()
    x[:110, :2] = 0.5 + 2.7 * dp * np.random.default_rng(5).random((110, 2))
    c["x"] = np.ascontiguousarray(x)
    _check(c)
