"""The folded passes on the CPU: the CTA programs of pstd_fold.cuh, emulated
thread by thread, against direct FP64 sums (fold_emulation.cu)."""
import os
import re
import subprocess

import pytest

from paper_2005_00322_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_folded_passes_match_direct_sums(tmp_path):
    """Derivatives in both directions, the second-order pass, and one leapfrog
    pass through the velocity's spectrum and back, for lengths on compiled and
    run-time radices, the four wall pairs, contiguous and strided lines with
    ragged tiles.  A transform of length L rounds each value about 3 log2(L)
    times (butterflies, twiddles), at most 33 roundings of 6e-8 in random
    directions: 3.4e-7 at L = 2048; 1e-6 leaves room for the four transforms
    of the second-order and conversion chains."""
    try:
        cc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    exe = str(tmp_path / "fold_emulation")
    r = subprocess.run([cc, *build.ARCH, "-O1", "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC,
                        os.path.join(HERE, "fold_emulation.cu"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr
    m = re.search(r"(\d+) checks, worst ([0-9.e+-]+), (\d+) without schedule", out.stdout)
    assert m, out.stdout[-2000:]
    assert int(m.group(1)) > 1000 and float(m.group(2)) < 1e-6, out.stdout[-2000:]
