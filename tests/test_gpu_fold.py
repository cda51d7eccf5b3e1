"""The folded passes on the GPU (schedule variant 6) against the FP64 oracle.

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


def rel(a, ref):
    a = a.detach().cpu().numpy().astype(np.float64)
    return float(np.linalg.norm(a - ref) / np.linalg.norm(ref))


def one_step(ncells, bcs, schedule=None):
    from paper_2005_00322_gb300 import Solver
    dt = pstd.dt_from_cfl(0.25 / np.sqrt(len(ncells)), DX, 1500.0)
    s = Solver(ncells, DX, bcs, dt=dt, schedule=schedule)
    od = pstd.Desc(ncells, (DX,), bcs, dt=dt)
    p0 = inputs.random_field(s.shapes[0], 1).astype(np.float32).astype(np.float64)
    u0 = [inputs.random_field(sh, 2 + i).astype(np.float32).astype(np.float64) * 1e-6
          for i, sh in enumerate(s.shapes[1:])]
    p = torch.tensor(p0.astype(np.float32), device="cuda")
    us = [torch.tensor(u.astype(np.float32), device="cuda") for u in u0]
    s.step(p, us)
    torch.cuda.synchronize()
    ref = pstd.step(od, pstd.State(p0, u0))
    return s, [rel(p, ref.p)] + [rel(u, r) for u, r in zip(us, ref.u)]


# one length for each radix of the combination (4, 6, 8, 10, 12, 16, 18, 20), run-time
# schedules (7, 11 and 13 as factors; 8 and 9 cells), odd and even outer and
# inner extents, every wall pair
@pytest.mark.parametrize("ncells,bcs", [
    ((32, 24), [("D", "D"), ("N", "N")]), ((54, 27), [("N", "D"), ("D", "N")]),
    ((64, 45), [("N", "N"), ("D", "D")]), ((75, 50), [("D", "N"), ("N", "D")]),
    ((486, 10), [("D", "D"), ("N", "D")]), ((9, 648), [("N", "N"), ("N", "N")]),
    ((729, 8), [("D", "N"), ("D", "D")]), ((1000, 9), [("N", "N"), ("D", "N")]),
    ((70, 77), [("D", "D"), ("N", "N")]), ((52, 91), [("N", "D"), ("D", "N")]),
    ((1024, 5), [("N", "D"), ("N", "N")]), ((24, 96, 18), [("D", "N"), ("N", "N"), ("D", "D")]),
    ((40, 36, 30), [("N", "N"), ("D", "D"), ("N", "D")]),
])
def test_step_on_every_radix(ncells, bcs):
    s, errs = one_step(ncells, bcs)
    # (extensions shorter than 16, N < 8, keep their other route)
    assert all(sc[0] == 6 for sc, n in zip(s.schedule(), ncells) if n >= 8), s.schedule()
    assert max(errs) < 1e-5, errs
    s.close()


@pytest.mark.parametrize("pairs", [1, 2, 4, 8])
def test_line_pairs_per_cta(pairs):
    """Compiled and run-time pairs per CTA, tiles with one to three lines left over."""
    s, errs = one_step((64, 33, 50), [("D", "D"), ("N", "N"), ("N", "D")], schedule=[(6, pairs)] * 3)
    assert [sc[2] for sc in s.schedule()] == [pairs] * 3
    assert max(errs) < 1e-5, errs
    s.close()


@pytest.mark.parametrize("n,bc", [(100, ("N", "N")), (256, ("D", "D")), (375, ("N", "D")), (512, ("D", "N"))])
def test_line_run_in_one_launch(n, bc):
    """A 1-D run loops over its steps in one kernel: the bits of single-pass
    launches (a batch member's), and the oracle's pressure."""
    from paper_2005_00322_gb300 import Solver
    from paper_2005_00322_gb300.batch import Batch
    dt = pstd.dt_from_cfl(0.2, DX, 1500.0)
    s = Solver((n,), DX, [bc], dt=dt)
    p0 = inputs.random_field(s.shapes[0], 5).astype(np.float32)
    p, u = torch.tensor(p0, device="cuda"), torch.zeros(s.shapes[1], device="cuda")
    s.init_velocity(p, [u])
    s.run(p, [u], 50)
    assert s.last_launch_count() == 3          # the run and the two velocity conversions
    b = Batch([dict(ncells=(n,), dx=DX, bc=[bc], dt=dt)])
    q, v = torch.tensor(p0, device="cuda"), torch.zeros(s.shapes[1], device="cuda")
    b.init_velocity([(q, [v])])
    b.run([(q, [v])], 50)
    b.sync()
    s.sync()
    assert torch.equal(p, q) and torch.equal(u, v)
    od = pstd.Desc((n,), (DX,), [bc], dt=dt)
    p064 = p0.astype(np.float64)
    ref = pstd.run(od, pstd.State(p064, pstd.init_velocity(od, p064, None, "halfstep")), 50)
    assert rel(p, ref.p) < 1e-4 and rel(u, ref.u[0]) < 1e-4
    s.close()
    b.close()
