"""The constants of the scaled interpolation operators (paper_2301_05985_gb300/csrc/lane_ops.cuh)
against 50 digits.  Every axis of the interpolation and of the tests multiplies by them, so an
error of a unit in the last place becomes several of the operators' results: each must be the
closest double."""
import os
import shutil
import subprocess
from decimal import Decimal, getcontext

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_constants_are_the_closest_doubles(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "lane_const_check")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(ROOT, "paper_2301_05985_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "lane_const_check.cu"), "-o", exe], check=True, capture_output=True)
    got = [float.fromhex(t) for t in subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split()]
    getcontext().prec = 50
    g = 1 / Decimal(3).sqrt()
    a, rho = (1 + g) / 2, (1 - g) / (1 + g)
    assert got == [float(rho)] + [float(a**n) for n in range(7)]
