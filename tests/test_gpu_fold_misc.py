"""Compiled derivatives and velocity conversions of the folded passes: the bits
of the run-time radices, which other line pairs per CTA select."""
import pytest
import torch

pytestmark = pytest.mark.gpu
DX = 1e-4
PAIRS = [("N", "N"), ("D", "D"), ("N", "D"), ("D", "N")]


# every length 2^k and 3 2^k with a compiled schedule, few and many lines, ragged tiles on both layouts
@pytest.mark.parametrize("n", [32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024])
@pytest.mark.parametrize("lines", [13, 1500])
@pytest.mark.parametrize("walls", PAIRS)
@pytest.mark.parametrize("axis", [0, 1])
def test_bits_of_the_run_time_radices(n, lines, walls, axis):
    from paper_2005_00322_gb300 import Solver
    ncells, bcs = [lines, lines], [("N", "N"), ("N", "N")]
    ncells[axis], bcs[axis] = n, walls
    out = []
    # pairs that are compiled for none of these schedules
    other = [(6, 1), None] if axis == 0 else [None, (6, 2 if n < 384 else 4)]
    for schedule in (None, other):
        s = Solver(tuple(ncells), DX, bcs, cfl=0.1, schedule=schedule)
        assert s.schedule()[axis][0] == 6
        g = torch.Generator().manual_seed(n)
        p, *us = [torch.randn(sh, generator=g).cuda() for sh in s.shapes]
        us = [1e-6 * u for u in us]
        res = [s.grad(axis, 0, p), s.grad(axis, 1, us[axis])]
        s.init_velocity(p, us)
        s.step(p, us)                 # conversions around one step
        s.sync()
        out.append(res + [p] + us)
        s.close()
    assert all(torch.equal(x, y) for x, y in zip(*out))
