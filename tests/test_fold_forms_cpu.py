"""Forms of the folded passes on the CPU that fold_emulation.cu's own run does
not tell apart (test_fold_cpu.py has the lengths and modes)."""
import os
import re
import subprocess

import pytest

from paper_2005_00322_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    """The lines that fold_emulation.cu's checks and then fold_accumulator.cu's print."""
    try:
        cc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    exe = str(tmp_path_factory.mktemp("emulation") / "emulation")
    r = subprocess.run([cc, *build.ARCH, "-O1", "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC, "-I", HERE,
                        os.path.join(HERE, "fold_accumulator.cu"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    return subprocess.run([exe], capture_output=True, text=True, timeout=300).stdout.splitlines()


def test_leapfrog_pass_takes_any_accumulator(lines):
    """A compiled pass adds onto the accumulator it is given, which on
    contiguous lines is p itself only on the last axis: not where the later
    axes store one node.  Both sides run the same operations but the order in
    which the compiler may fuse the last addition: one rounding (6e-8)."""
    m = re.fullmatch(r"(\d+) compared, (\d+) failed", lines[-1])
    assert m and int(m.group(1)) > 500 and int(m.group(2)) == 0, lines[-20:]


def test_no_check_fails_on_any_value(lines):
    """Every check of fold_emulation.cu that is not below its bound prints a line
    of its own, a NaN (which its largest error passes over) included."""
    assert [x for x in lines if not re.fullmatch(r"\d+ checks, worst \S+, \d+ without schedule|\d+ compared, \d+ failed",
                                                 x)] == []
