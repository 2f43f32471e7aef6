"""The load and the read-back of a state from every kind of memory (pageable
and page-locked host memory, device memory, and mixtures within one call):
the same bits in, the same bits out; and the reference sums of layouts whose
warps hold one, a few and many different (h, m)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2411_13992_gb300 as sph
from paper_2411_13992_gb300 import cases

pytestmark = pytest.mark.gpu

KINDS = ("pageable", "pinned", "device")


def _as(a, kind):
    if kind == "pageable":
        return np.array(a)
    t = torch.from_numpy(np.array(a))
    return t.pin_memory() if kind == "pinned" else t.cuda()


def _pick(mix, k):
    return mix[k % len(mix)]


def _case(dim):
    c = cases.cavity2d(21, jitter_dp=0.1) if dim == 2 else cases.tgv3d(9, jitter_dp=0.1)
    rng = np.random.default_rng(3)
    ad = [rng.standard_normal((c["n"], 3)) for _ in range(2)]
    for a in ad:
        a[c["kind"] != 0] = 0.0
        a[:, dim:] = 0.0
    return c, ad


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("mix", [("pageable",), ("pinned",), ("device",), ("device", "pageable"),
                                 ("pageable", "device", "pinned"), ("pinned", "pageable", "device", "device")])
def test_state_in_and_out(precision, dim, mix):
    c, (a, dr) = _case(dim)
    n = c["n"]
    real = np.float32 if precision == 32 else np.float64
    sim = sph.Simulation(c, precision=precision)
    try:
        args = [c["x"], c["v"], a, dr, c["h"], c["m"], c["kind"], c["vw"]]
        sph.sph_set_state(sim.ctx, *[_as(q, _pick(mix, k)) for k, q in enumerate(args)])
        sim.build_cells()
        outs = [_as(np.full((n, 3), 7.0), _pick(mix, k + 1)) for k in range(4)] + [_as(np.full(n, 7.0), mix[0])]
        sph.sph_get_state(sim.ctx, *outs)
        sim.sync()
        got = [o if isinstance(o, np.ndarray) else o.cpu().numpy() for o in outs]
        v = np.where((c["kind"] != 0)[:, None], c["vw"], c["v"])
        keep = np.arange(3) < dim
        for g, want in zip(got[:4], (c["x"], v.astype(real), a.astype(real), dr.astype(real))):
            assert np.array_equal(g, np.where(keep, want.astype(np.float64), 0.0))
        one = np.full((n, 3), 7.0)          # a single output, the others not asked for
        sph.sph_get_state(sim.ctx, None, one)
        assert np.array_equal(one, got[1])
    finally:
        sim.close()


@pytest.mark.parametrize("distinct", [1, 2, 4, 5, 40])
@pytest.mark.parametrize("dim", [2, 3])
def test_reference_sums_of_mixed_resolutions(dim, distinct):
    """sigma0 of the density sum (Eq. 8) for 1 to 40 different h, interleaved
    so that a warp holds all of them: rho against the oracle's, whose sigma0
    is the plain lattice sum (FP64 bound of the parity tests)."""
    c = dict(cases.tgv2d(24, jitter_dp=0.1) if dim == 2 else cases.tgv3d(10, jitter_dp=0.1))
    n = c["n"]
    c["h"] = c["h"] * (1.0 + 0.15 * (np.arange(n) % distinct) / max(distinct - 1, 1))
    c["m"] = c["m"] * (1.0 + 0.01 * (np.arange(n) % distinct))
    c["h_min"], c["h_max"] = float(c["h"].min()), float(c["h"].max())
    P = oracle.make_params(c["dim"], c["lo"], c["L"], c["periodic"], c["rho0"], c["c"], c["eta"], c["h_min"],
                           u_ref=c["u_ref"])
    ref = oracle.force_pass(P, c, c["x"], c["v"], oracle.sigma0_for(c, dim))["rho"]
    sim = sph.Simulation(c, precision=64)
    try:
        sim.set_state()
        sim.build_cells()
        rho = sim.get_state()["rho"]
        sim.sync()
    finally:
        sim.close()
    assert np.abs(rho - ref).max() <= 1e-12 * np.abs(ref).max()
