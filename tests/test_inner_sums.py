"""The running sum of the inner solve's FP32 dot products (paper_2301_05985_gb300/csrc/dot4.cuh)
rounds once per four products at its own size.

Bound on the mean square error of sums of positive terms: a rounding is off by ulp / sqrt 12 in
the mean, and ulp(s) <= 2^-23 s, so the sum of c steps s_1 .. s_c is off by at most
2^-23 / sqrt 12 sqrt(s_1^2 + .. + s_c^2); the three roundings inside a step are at sums of one to
three products, below a fifth of s_1 .. s_c in all (10 % on the bound).  A chain of four fused
operations per step has four such roundings a step: twice that and more."""
import math
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("chunks", [6, 43, 171])
def test_running_sum_rounds_once_per_float4(chunks, tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "dot4_check")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-Xcompiler", "-ffp-contract=off",
                    "-I", os.path.join(ROOT, "paper_2301_05985_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "dot4_check.cu"), "-o", exe], check=True, capture_output=True)
    out = subprocess.run([exe, "4000", str(chunks)], capture_output=True, text=True, check=True).stdout.split("\n")
    err = bound = 0.0
    for line in out[:4000]:
        s, exact, sq = (float.fromhex(t) for t in line.split())
        err += (s - exact) ** 2
        bound += sq * 2.0**-46 / 12
    assert math.sqrt(err) <= 1.1 * math.sqrt(bound)
