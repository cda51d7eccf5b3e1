"""Cooperative runs on folded schedules: the bits of the per-axis launches."""
import itertools

import pytest
import torch

pytestmark = pytest.mark.gpu
DX = 1e-4
PAIRS = [("N", "N"), ("D", "D"), ("N", "D"), ("D", "N")]


def filled(shapes, seed):
    g = torch.Generator().manual_seed(seed)
    p, *us = [torch.randn(sh, generator=g).cuda() for sh in shapes]
    return p, [1e-6 * u for u in us]


def copy(f):
    return f[0].clone(), [u.clone() for u in f[1]]


def same(a, b):
    return torch.equal(a[0], b[0]) and all(torch.equal(x, y) for x, y in zip(a[1], b[1]))


# compiled schedules (ragged tiles on either layout, more and fewer lines than the
# grid's CTAs take, many and few lines' pairs), run-time radices (70, 9)
@pytest.mark.parametrize("ncells", [(24, 24), (50, 50), (81, 81), (100,), (1000,), (33, 33), (45, 45, 45), (64, 64, 64),
                                    (384, 384), (1024, 1024),
                                    (128, 128, 128), (48, 48, 48), (70, 70), (9, 9, 9)])
def test_single(ncells):
    from paper_2005_00322_gb300 import Solver
    bcs = [PAIRS[(i + len(ncells)) % 4] for i in range(len(ncells))]
    runs = []
    for persistent in (False, True):
        s = Solver(ncells, DX, bcs, cfl=0.1, persistent=persistent)
        f = filled(s.shapes, 3)
        s.run(*f, 20)                # below a graph's block: one pass after the other
        s.sync()
        assert s.persistent()[0] == (persistent and all(v[0] == 6 for v in s.schedule()))
        runs.append(f)
        s.close()
    assert same(*runs)


@pytest.mark.parametrize("ncells,count", [((90, 90), 16), ((27, 27, 27), 7), ((100,), 40), ((256,), 400), ((48, 48), 16), ((64, 64, 64), 3),
                                          ((77, 77), 3)])
def test_batch(ncells, count):
    from paper_2005_00322_gb300.batch import Batch
    walls = list(itertools.islice(itertools.cycle(itertools.product(PAIRS, repeat=len(ncells))), count))
    b = Batch([dict(ncells=ncells, dx=DX, bc=list(w), cfl=0.1) for w in walls])
    assert b.persistent_kind() == "register"
    start = [filled(sh, m) for m, sh in enumerate(b.shapes)]
    graph, coop = [copy(f) for f in start], [copy(f) for f in start]
    b.run(graph, 20)
    b.sync()
    b.set_persistent(True)
    b.run(coop, 20)
    b.sync()
    assert all(same(x, y) for x, y in zip(graph, coop))
    b.close()
