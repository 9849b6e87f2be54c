"""The products of the block fixed-point transforms (csrc/fft_fx.cuh), compiled for the host: within
two units of the exact product and on average within 0.6, for every twiddle constant, for the constants whose
cross terms are largest (high word near one third, low word near 2^31) and for stored symbol values, over
the accepted range of x (tests/c/fx_products.cpp)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_products_stay_within_two_units_and_have_no_errors_of_one_sign(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "fx_products")
    r = subprocess.run([cxx, "-std=c++17", "-O1", os.path.join(HERE, "c", "fx_products.cpp"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
