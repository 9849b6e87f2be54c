"""That the grids of test_gpu_paired_wave.py are what it takes them for on this device: pairs of CTAs on
the last wave of (4, 4, 4), (5, 4, 8) and (6, 4, 9) x points, one CTA per x point on its reference of
(4, 4, 9) (tests/c/paired_plan.cu asks the library's own plan)."""
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_the_paired_grids_are_paired_and_the_reference_is_not(tmp_path):
    import paper_2205_02380_gb300 as pkg
    from paper_2205_02380_gb300 import build as B
    pkg.chasm.lib()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    exe = str(tmp_path / "paired_plan")
    r = subprocess.run([B.nvcc(), *B.ARCH, "-std=c++17", "-cudart", "shared",
                        os.path.join(HERE, "c", "paired_plan.cu"), "-L", B.HERE, "-lchasm",
                        "-Xlinker", "-rpath=" + B.HERE, "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    paired, single = [4 * 4 * 4, 5 * 4 * 8, 6 * 4 * 9], [4 * 4 * 9, sms]
    r = subprocess.run([exe, *map(str, paired + single)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    plan = {int(a): (int(b), int(c)) for a, b, c in (line.split() for line in r.stdout.splitlines())}
    assert [plan[n][0] for n in paired] == [2, 2, 2]
    assert plan[64][1] == 128 and plan[160][1] == plan[216][1] == sms
    assert [plan[n] for n in single] == [(1, 144), (1, sms)]
