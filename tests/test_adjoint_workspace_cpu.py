"""Size of the FP64 adjoint's workspace: the tape holds its steps' neighbour
lists while they take at most 1 GiB together; beyond that a tape slot takes
what its forward values take (the reverse sweep builds the lists again)."""
import pytest

import paper_2411_13992_gb300 as sph
from paper_2411_13992_gb300 import cases

GIB = 1 << 30


def _grow(c, n, steps):
    size = []
    for k in (0, steps):
        p = sph.params_from_case(c, 64)
        p.adjoint_steps = k
        size.append(sph.sph_query_workspace(p, n))
    return size[1] - size[0]


# forward values of a slot, bytes a particle: id and cell 4 each, kind 1, h, m, sigma0 8 each, velocity record 32, x and
# R 8 a component each; the cell starts 4 a cell at most as many as particles; cotangents and scratch of the sweep, for
# all slots together, at most 300 bytes a particle
@pytest.mark.parametrize("case,values", [(lambda: cases.tgv2d(16), 4 + 4 + 1 + 24 + 32 + 32 + 4),
                                         (lambda: cases.tgv3d(16), 4 + 4 + 1 + 24 + 32 + 48 + 4)])
def test_a_large_tape_holds_no_lists(case, values):
    c = case()
    n, steps = 1_000_000, 200
    assert _grow(c, n, steps) <= n * (values * steps + 300) + (steps + 20) * 16 * 256


@pytest.mark.parametrize("case,cap", [(lambda: cases.tgv2d(16), 96), (lambda: cases.tgv3d(16), 128)])
def test_a_small_tape_holds_its_lists(case, cap):
    c = case()
    slot = 4 * c["n"] * (cap + 1)
    held = GIB // slot
    assert _grow(c, c["n"], held) >= held * slot
    assert _grow(c, c["n"], held + 1) < held * slot
