"""The constants of the scaled interpolation operators (paper_2301_05985_gb300/csrc/lane_ops.cuh)
against 50 digits.  Every axis of the interpolation and of the tests multiplies by them, so an
error of a unit in the last place becomes several of the operators' results: each must be the
closest double.  An FP32 product with one rounds once: half a unit in the last place, 2^-24
relative, and 2^-46 for the low part of the constant."""
import os
import random
import shutil
import subprocess
from decimal import Decimal, getcontext
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
getcontext().prec = 50


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path_factory.mktemp("lane") / "lane_const_check")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(ROOT, "paper_2301_05985_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "lane_const_check.cu"), "-o", exe], check=True, capture_output=True)
    return lambda text: [float.fromhex(t) for t in subprocess.run([exe], input=text, capture_output=True, text=True,
                                                                  check=True).stdout.split()]


def _a():
    return (1 + 1 / Decimal(3).sqrt()) / 2


def test_constants_are_the_closest_doubles(driver):
    g = 1 / Decimal(3).sqrt()
    assert driver("") == [float((1 - g) / (1 + g))] + [float(_a()**n) for n in range(7)]


def test_fp32_products_round_once(driver):
    rng = random.Random(3)
    ops = [(float(np.float32(rng.choice([-1, 1]) * 10.0**rng.uniform(-12, 6))), rng.randint(1, 6), rng.randint(-24, 24))
           for _ in range(4000)]
    got = driver("\n".join(f"{x.hex()} {n} {e}" for x, n, e in ops) + "\n")[8:]
    bound = Fraction(1, 2**24) + Fraction(1, 2**46)
    for (x, n, e), y in zip(ops, got):
        exact = Fraction(x) * Fraction(_a()**n) * Fraction(2)**e
        assert abs(Fraction(y) - exact) <= bound * abs(exact), (x, n, e)
