"""Forms of the folded passes on the CPU that fold_emulation.cu's own run does
not tell apart (test_fold_cpu.py has the lengths and modes)."""
import os
import re
import subprocess

import pytest

from paper_2005_00322_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def run(src, tmp_path):
    try:
        cc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    exe = str(tmp_path / "emulation")
    r = subprocess.run([cc, *build.ARCH, "-O1", "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC, "-I", HERE,
                        os.path.join(HERE, src), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    return subprocess.run([exe], capture_output=True, text=True, timeout=300)


def test_leapfrog_pass_takes_any_accumulator(tmp_path):
    """A compiled pass adds onto the accumulator it is given, which on
    contiguous lines is p itself only on the last axis: not where the later
    axes store one node.  Both sides run the same operations but the order in
    which the compiler may fuse the last addition: one rounding (6e-8)."""
    r = run("fold_accumulator.cu", tmp_path)
    m = re.search(r"(\d+) compared, (\d+) failed", r.stdout)
    assert m, r.stdout[-2000:]
    assert r.returncode == 0 and int(m.group(1)) > 500 and int(m.group(2)) == 0, r.stdout[-2000:]
