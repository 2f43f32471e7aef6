"""sph_density_noalloc with per-particle constants that do not lie on their
natural alignment (views into a packed byte buffer): the same bits as from
aligned arrays."""
import numpy as np
import pytest
import torch

import oracle
import paper_2411_13992_gb300 as sph
from paper_2411_13992_gb300 import cases

pytestmark = pytest.mark.gpu


def _shifted(a, by):
    """The bytes of ``a`` on the device, ``by`` bytes past an aligned address."""
    raw = torch.from_numpy(np.frombuffer(a.tobytes(), np.uint8).copy())
    buf = torch.zeros(raw.numel() + 16, dtype=torch.uint8, device="cuda")
    view = buf[by:by + raw.numel()]
    view.copy_(raw)
    assert view.data_ptr() % 8 == by
    return view


@pytest.mark.parametrize("by", [1, 4])
def test_noalloc_constants_off_their_alignment(by):
    c = cases.cylinder2d(res=3, box=(12.0, 8.0), center=(4.0, 4.0), refine=(3.0, 9.0, 2.5, 5.5))
    p = sph.params_from_case(c, 64)
    s0 = oracle.sigma0_for(c, 2)
    x = torch.from_numpy(np.array(c["x"])).cuda()
    st = torch.cuda.current_stream().cuda_stream
    rho = {}
    for shift in (0, by):
        h, m, kind, s = (_shifted(np.ascontiguousarray(c[k]), shift) if k else _shifted(s0, shift)
                         for k in ("h", "m", "kind", None))
        for given in (None, s):
            out = torch.full((c["n"],), float("nan"), dtype=torch.float64, device="cuda")
            sph.sph_density_noalloc(p, c["n"], x, h, m, kind, given, out, st)
            torch.cuda.synchronize()
            rho[shift, given is not None] = out.cpu().numpy()
    for given in (False, True):
        assert np.isfinite(rho[0, given]).all()
        assert np.array_equal(rho[0, given], rho[by, given])
