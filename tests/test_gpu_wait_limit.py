"""The waits of the double-precision Coulomb kernel (csrc/group_bar.cuh) end: with a partner at
once; without one after the given number of tries, the later waits of the block after one try, and the
default limit after about a second (tests/c/wait_limit.cu).  The words that a wait sets when it runs out
are what the kernel turns into NaN and the status of chasm_moments."""
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_a_wait_that_nobody_ends_runs_out_once(tmp_path):
    from paper_2205_02380_gb300 import build as B
    exe = str(tmp_path / "wait_limit")
    r = subprocess.run([B.nvcc(), *B.ARCH, "-std=c++17", "-O3", os.path.join(HERE, "c", "wait_limit.cu"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    rows = [tuple(int(v) for v in line.split()) for line in r.stdout.splitlines()]
    assert len(rows) == 5
    for partner, tries, ran_out, first, later in rows:
        if partner:
            assert ran_out == 0
        else:
            assert ran_out == 3           # both words
            assert first > 8 * later      # 64 tries or more, then one (two where the first stands apart)
    assert 0.3e9 < rows[-1][3] < 3e9
