"""The FP32 force pass at the grid size where its software pipeline deepens (at
most four blocks of 128 particles per SM), and lists shorter than the
pipeline: the step against the FP64 oracle within the FP32 tolerances of the
parity tests.  Particles far apart have no neighbours at all, a row of them
one or two."""
import numpy as np
import pytest
import torch

import oracle
import paper_2411_13992_gb300 as sph
from paper_2411_13992_gb300 import cases

from gpu_helpers import compare_step, oracle_params

pytestmark = pytest.mark.gpu


def _check(c):
    oracle.set_threads(16)
    P = oracle_params(c)
    s0 = oracle.sigma0_for(c, c["dim"])
    fp = oracle.force_pass(P, c, c["x"], c["v"], s0)
    state = {"x": c["x"], "v": c["v"], "a": fp["a"], "dr": fp["dr"]}
    err, _, _ = compare_step(c, state, oracle.time_step(P, c["v"], c["kind"]), s0, P, precision=32)
    for k in ("x", "v", "rho"):
        assert err[k] <= 1e-5, err
    assert err["a"] <= 1e-3, err


@pytest.mark.parametrize("off", [-1, 0, 1])
@pytest.mark.parametrize("dim", [2, 3])
def test_both_sides_of_the_line(dim, off):
    n = torch.cuda.get_device_properties(0).multi_processor_count * 4 * 128 + off
    side = int(np.ceil(n ** (1.0 / dim) - 1e-9))
    c = dict((cases.tgv2d if dim == 2 else cases.tgv3d)(side, jitter_dp=0.1, seed=7))
    for k in ("x", "v", "h", "m", "kind", "vw"):
        c[k] = np.ascontiguousarray(c[k][:n])
    c["n"] = n
    _check(c)


@pytest.mark.parametrize("per_group", [1, 2, 3, 4, 5, 6, 7, 9, 10, 11, 12])
def test_lists_shorter_than_the_pipeline(per_group):
    """Groups of 1 to 12 particles within one smoothing length, the groups out
    of each other's reach: lists of 0 to 11 entries around the pipeline's 5 and 10."""
    c = dict(cases.tgv2d(40))
    rng = np.random.default_rng(per_group)
    dp = c["dp"]
    centres = np.stack(np.meshgrid(np.arange(5), np.arange(5)), -1).reshape(-1, 2) * 8.0 * dp + 3.0 * dp
    pts = centres[:, None, :] + (rng.random((len(centres), per_group, 2)) - 0.5) * 1.2 * dp
    n = pts.shape[0] * per_group
    c["x"] = np.zeros((n, 3))
    c["x"][:, :2] = pts.reshape(n, 2)
    for k in ("v", "h", "m", "kind", "vw"):
        c[k] = np.ascontiguousarray(c[k][:n])
    c["v"] = rng.standard_normal((n, 3)) * np.array([1.0, 1.0, 0.0])
    c["n"] = n
    _check(c)
