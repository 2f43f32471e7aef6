"""The graph of eight steps (calls of 16 steps or more), captured behind steps of
the short graph: from both parities of the state sets, with the graph of two
steps and a direct step for the rest of a call, after a change of viscosity that
drops the graphs, and with graphs captured before any sort has run; states,
diagnostics and launch counts are those of direct launches."""
import numpy as np
import pytest
import torch

import paper_2411_13992_gb300 as sph
from paper_2411_13992_gb300 import cases

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    assert torch.cuda.is_available()


def _run(c, precision, graphs, plan, ad=None):
    sim = sph.Simulation(c, precision=precision, graphs=graphs)
    out = []
    try:
        sim.set_state(a=None if ad is None else ad[0], dr=None if ad is None else ad[1])
        sim.build_cells()
        for what, arg in plan:
            l0 = sim.launches()
            if what == "eta":
                sph.sph_set_eta(sim.ctx, arg * c["eta"])
            else:
                sim.step(arg)
                out.append((sim.get_state(), sim.diag(), sim.launches() - l0))
        assert sim.sync() is None
        return out
    finally:
        sim.close()


# (an odd number of steps changes the parity of the state sets)
PLANS = {
    "long_call_first": [("step", 40), ("step", 17), ("step", 19), ("step", 40)],
    "shortest_calls": [("step", 16), ("step", 16), ("step", 15), ("step", 17), ("step", 1), ("step", 23)],
    "short_graph_first": [("step", 3), ("step", 2), ("step", 19), ("step", 27), ("step", 18)],
    "viscosity": [("step", 20), ("eta", 2.0), ("step", 16), ("step", 1), ("step", 27), ("eta", 1.5), ("step", 19)],
}


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("case", ["tgv2d", "cavity", "tgv3d"])
@pytest.mark.parametrize("plan", sorted(PLANS))
@pytest.mark.parametrize("ad_given", [False, True])
def test_long_graphs_are_bit_identical(precision, case, plan, ad_given):
    c = {"tgv2d": cases.tgv2d(20), "cavity": cases.cavity2d(16), "tgv3d": cases.tgv3d(8)}[case]
    ad = None
    if ad_given:                     # the first sort then lies inside the first capture
        rng = np.random.default_rng(8)
        ad = [1e-3 * rng.standard_normal((c["n"], 3)), 1e-3 * c["dp"] * rng.standard_normal((c["n"], 3))]
        for q in ad:
            q[:, c["dim"]:] = 0.0
            q[c["kind"] != 0] = 0.0
    on, off = (_run(c, precision, g, PLANS[plan], ad) for g in (1, 0))
    for k, ((s1, d1, l1), (s0, d0, l0)) in enumerate(zip(on, off)):
        for q in ("x", "v", "a", "dr", "rho"):
            assert np.isfinite(s1[q]).all() and np.array_equal(s1[q], s0[q]), (k, q)
        assert d1["ke"] == d0["ke"] and d1["dt_next"] == d0["dt_next"] and d1["steps"] == d0["steps"], k
        assert l1 == l0, k
