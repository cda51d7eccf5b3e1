"""2-D runs with both axis passes of a step side by side: the bits of one pass
after the other (a batch member's launches), and the state a plan is left in."""
import subprocess
import sys

import pytest
import torch

pytestmark = pytest.mark.gpu
DX = 1e-4
BLOCK = 32


def filled(shapes, seed):
    g = torch.Generator().manual_seed(seed)
    p, *us = [torch.randn(sh, generator=g).cuda() for sh in shapes]
    return p, [1e-6 * u for u in us]


# one block, blocks with and without a tail; ragged tiles; every wall pair on either axis
@pytest.mark.parametrize("ncells,bcs,steps", [
    ((512, 512), [("D", "D"), ("N", "N")], 64), ((375, 300), [("N", "D"), ("D", "N")], 95),
    ((64, 48), [("N", "N"), ("D", "D")], 32), ((1000, 24), [("D", "N"), ("N", "D")], 70),
    ((24, 1000), [("D", "D"), ("D", "N")], 33), ((81, 135), [("N", "N"), ("N", "D")], 128),
])
def test_bits_of_sequential_passes(ncells, bcs, steps):
    from paper_2005_00322_gb300 import Solver
    from paper_2005_00322_gb300.batch import Batch
    s, b = Solver(ncells, DX, bcs, cfl=0.1), Batch([dict(ncells=ncells, dx=DX, bc=bcs, cfl=0.1)])
    p, us = filled(s.shapes, 1)
    q, vs = p.clone(), [u.clone() for u in us]
    for _ in range(2):                 # the second run replays the recorded block
        s.run(p, us, steps)
        b.run([(q, vs)], steps)
    s.sync()
    b.sync()
    # two passes a step, the sum of the two fields after each block, two conversions per axis
    assert s.last_launch_count() == 2 * steps + steps // BLOCK + 4
    assert torch.equal(p, q) and all(torch.equal(u, v) for u, v in zip(us, vs))
    s.close()
    b.close()


def test_a_captured_run_decides_nothing():
    """A run of a block or more cannot be captured (it records a graph itself);
    the plan's later runs still go side by side."""
    code = """
import torch
from paper_2005_00322_gb300 import Solver
s = Solver((64, 48), 1e-4, [("N", "N"), ("D", "D")], cfl=0.1)
p, us = s.zeros()
torch.cuda.synchronize()
try:
    with torch.cuda.graph(torch.cuda.CUDAGraph()):
        s.run(p, us, 64)
    print("captured")
except Exception as e:
    print("refused")
torch.cuda.synchronize()
s.run(p, us, 64)
s.sync()
print(s.last_launch_count())
"""
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=120)
    assert r.stdout.split() == ["refused", str(2 * 64 + 2 + 4)], (r.stdout, r.stderr[-2000:])
