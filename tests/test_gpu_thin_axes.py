"""Grids whose trailing axes store a single pressure node (one cell with one
Dirichlet wall, two cells between Dirichlet walls), so that an axis before the
last is contiguous too, against the FP64 oracle.

Tolerances are those of the plain path: 1e-5 relative L2 for one step, 1e-4
for a run.
"""
import numpy as np
import pytest
import torch

from oracle import pstd
from paper_2005_00322_gb300 import inputs

pytestmark = pytest.mark.gpu
DX = 1e-4
STEPS = 50

# compiled folded lengths, a run-time one (70 = 2 5 7), a convolution line (67), a register line (6)
GRIDS = [
    ((256, 2), [("N", "N"), ("D", "D")]),
    ((64, 1), [("N", "N"), ("N", "D")]),
    ((100, 1), [("D", "N"), ("D", "N")]),
    ((512, 2), [("N", "D"), ("D", "D")]),
    ((40, 36, 2), [("N", "N"), ("D", "D"), ("D", "D")]),
    ((64, 32, 1), [("D", "N"), ("N", "D"), ("N", "D")]),
    ((48, 2, 1), [("D", "D"), ("D", "D"), ("D", "N")]),
    ((70, 2), [("N", "N"), ("D", "D")]),
    ((67, 1), [("N", "N"), ("N", "D")]),
    ((6, 2), [("N", "N"), ("D", "D")]),
]


def rel(a, ref):
    a = a.detach().cpu().numpy().astype(np.float64)
    return float(np.linalg.norm(a - ref) / np.linalg.norm(ref))


def start(shapes, dtype=np.float32):
    p = inputs.random_field(shapes[0], 1).astype(dtype)
    # velocities of the size a pressure of order one drives (p / (rho0 c0))
    return p, [inputs.random_field(sh, 2 + i).astype(dtype) * dtype(1e-6) for i, sh in enumerate(shapes[1:])]


def on_gpu(p, us):
    return torch.tensor(p, device="cuda"), [torch.tensor(u, device="cuda") for u in us]


def oracle(ncells, bcs, dt, p, us, steps):
    od = pstd.Desc(ncells, (DX,), bcs, dt=dt)
    return pstd.run(od, pstd.State(p.astype(np.float64), [u.astype(np.float64) for u in us]), steps)


def time_step(ncells):
    return pstd.dt_from_cfl(0.25 / np.sqrt(len(ncells)), DX, 1500.0)


@pytest.mark.parametrize("ncells,bcs", GRIDS)
@pytest.mark.parametrize("persistent", [False, True])
def test_single(ncells, bcs, persistent):
    from paper_2005_00322_gb300 import Solver
    dt = time_step(ncells)
    s = Solver(ncells, DX, bcs, dt=dt, persistent=persistent)
    p0, u0 = start(s.shapes)
    p, us = on_gpu(p0, u0)
    s.step(p, us)
    s.sync()
    ref = oracle(ncells, bcs, dt, p0, u0, 1)
    assert max([rel(p, ref.p)] + [rel(u, r) for u, r in zip(us, ref.u)]) < 1e-5
    p, us = on_gpu(p0, u0)
    s.run(p, us, STEPS)
    s.sync()
    ref = oracle(ncells, bcs, dt, p0, u0, STEPS)
    assert rel(p, ref.p) < 1e-4
    s.close()


@pytest.mark.parametrize("cooperative", [False, True])
def test_batch(cooperative):
    from paper_2005_00322_gb300.batch import Batch
    b = Batch([dict(ncells=n, dx=DX, bc=w, dt=time_step(n)) for n, w in GRIDS])
    b.set_persistent(cooperative)
    host = [start(sh) for sh in b.shapes]
    fields = [on_gpu(*h) for h in host]
    b.run(fields, STEPS)
    b.sync()
    for (n, w), (p0, u0), (p, _) in zip(GRIDS, host, fields):
        assert rel(p, oracle(n, w, time_step(n), p0, u0, STEPS).p) < 1e-4, n
    b.close()


def test_autotuned():
    """The candidates of a contiguous axis before the last: its compiled pairs."""
    from paper_2005_00322_gb300 import Solver
    ncells, bcs = (48, 48, 2), [("N", "D"), ("D", "D"), ("D", "D")]
    s = Solver(ncells, DX, bcs, dt=time_step(ncells), autotune=True)
    variant, _, pairs, _ = s.schedule()[1]
    assert variant != 6 or pairs in (1, 8)
    p0, u0 = start(s.shapes)
    p, us = on_gpu(p0, u0)
    s.run(p, us, STEPS)
    s.sync()
    assert rel(p, oracle(ncells, bcs, time_step(ncells), p0, u0, STEPS).p) < 1e-4
    s.close()
