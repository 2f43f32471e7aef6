"""Invalid masses and smoothing lengths are reported by sph_sync as
SPH_ERR_INPUT, whatever the reference sum of Eq. 8 would be for them (a mass of
zero or an infinite h asks for a lattice without end), and leave the context
usable; the reference sum on both sides of the line from which it is taken at
its limit dp^-D."""
import numpy as np
import pytest
import torch

import paper_2411_13992_gb300 as sph
from paper_2411_13992_gb300 import cases

pytestmark = pytest.mark.gpu

ERR_INPUT = 8


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    assert torch.cuda.is_available()


BAD = [("m", 0.0), ("m", -1.0), ("m", -1e-30), ("m", np.nan), ("m", np.inf), ("h", 0.0), ("h", -1.0), ("h", -1e30),
       ("h", np.inf), ("h", np.nan), ("h", 0.99), ("h", 1.16)]


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("precision,variable", [(64, False), (64, True), (32, False), (32, True)])
def test_invalid_mass_or_h_is_reported(dim, precision, variable):
    c = dict((cases.tgv2d if dim == 2 else cases.tgv3d)(8, jitter_dp=0.1))
    if variable:
        c["h_max"] = 1.15 * c["h_max"]
    sim = sph.Simulation(c, precision=precision)
    try:
        for what, value in BAD:
            for at in (0, 7, c["n"] - 1):
                bad = {k: c[k].copy() for k in ("h", "m")}
                # h in units of the case's, a mass as it is
                bad[what][at] = value * c["h_min"] if what == "h" else value
                sph.sph_set_state(sim.ctx, c["x"], c["v"], None, None, bad["h"], bad["m"], c["kind"], c["vw"])
                with pytest.raises(sph.SphError) as e:
                    sim.sync()
                assert e.value.status == ERR_INPUT, (what, value, at)
                sim.build_cells()                   # runs to its end on it
                sph.sph_set_state(sim.ctx, c["x"], c["v"], None, None, c["h"], c["m"], c["kind"], c["vw"])
                sim.build_cells()
                try:
                    sim.sync()
                except sph.SphError:                # what the pass over the invalid state reported
                    pass
                rho = sim.get_state()["rho"]
                sim.sync()
                assert np.isfinite(rho).all() and np.abs(rho / c["rho0"] - 1.0).max() < 0.5, (what, value, at)
    finally:
        sim.close()


@pytest.mark.parametrize("dim,ratio", [(2, 499.0), (2, 501.0), (2, 1e9), (2, 1e60), (3, 99.0), (3, 101.0), (3, 1e60)])
def test_reference_sum_of_a_light_particle(dim, ratio):
    """A lone particle of h = ratio dp: rho = rho0 W(0) / sigma0, and sigma0
    dp^D is 1 within the limit's own difference (4e-14 at the line in 3-D, less
    in 2-D) and, below the line, the rounding of a sum of (2 ratio)^D terms."""
    h = 1.3
    dp = h / ratio
    c = {"name": "light", "dim": dim, "n": 1, "x": np.array([[4.0, 6.0, 5.0]]), "v": np.zeros((1, 3)),
         "h": np.full(1, h), "m": np.full(1, dp ** dim), "kind": np.zeros(1, np.int8), "vw": np.zeros((1, 3)),
         "lo": (0.0, 0.0, 0.0), "L": (20.0, 20.0, 20.0), "periodic": (0, 0, 0), "rho0": 1.0, "c": 10.0, "eta": 0.0,
         "g": (0.0, 0.0, 0.0), "h_min": h, "h_max": h, "u_ref": 0.4}
    sim = sph.Simulation(c, precision=64, fixed_dt=0.01)
    try:
        sim.set_state()
        sim.build_cells()
        assert sim.sync() is None
        rho = sim.get_state()["rho"][0]
    finally:
        sim.close()
    w0 = (7.0 / (4.0 * np.pi) if dim == 2 else 21.0 / (16.0 * np.pi)) / h ** dim
    terms = (2.0 * ratio + 1.0) ** dim if ratio < 600 else 0.0
    # rho is stored as rho - rho0: an absolute rounding of 2^-53 rho0 beside it
    tol = (1e-13 + terms * 2.0 ** -53) * w0 * dp ** dim + 2.0 ** -52
    assert abs(rho - w0 * dp ** dim) <= tol
