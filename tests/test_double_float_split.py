"""The integer split of a double into a double-float, its join, and the quick operations
(paper_2301_05985_gb300/csrc/df32.cuh), on the host, against exact rational arithmetic.

Bounds, with u = 2^-24: the split keeps 24 + 24 bits and a sign (2^-48 relative, normal
range of float), its join is exact to a rounding of FP64; the quick sum rounds the low
parts' sum, the error term and the renormalisation (at most 6 u^2 (|a| + |b|)), the quick
fused multiply-add the three low products as well (10 u^2 (|a b| + |c|))."""
import math
import os
import random
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from test_double_float import _df, _exact

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("dfs") / "df_split_check")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-Xcompiler", "-ffp-contract=off",
                    "-I", os.path.join(ROOT, "paper_2301_05985_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "df_split_check.cu"), "-o", out], check=True, capture_output=True)
    return out


def test_split_join_and_quick_operations(driver):
    rng = random.Random(7)
    xs = [0.0, -0.0, 1.0, -1.0, 3.0, 1.0 + 2.0**-52, 1.0 - 2.0**-53, 1.0 + 2.0**-24, 1.0 + 3 * 2.0**-25,
          2.0**-126, -(2.0**-126), 2.0**-140, 5e-324, 3.4028234663852886e38, -3.0e38, 1e39, math.inf, -math.inf, math.nan]
    for e in range(-100, 128):
        for m in (1.0, math.nextafter(1.0, 2.0), math.nextafter(2.0, 1.0), 1.0 + 2.0**-24 + 2.0**-52):
            x = math.ldexp(m, e - 1)
            xs += [x, -x]
    xs += [rng.choice([-1, 1]) * math.ldexp(rng.uniform(1.0, 2.0), rng.randint(-90, 120)) for _ in range(3000)]
    ops = []
    for i in range(len(xs)):
        sa, sb = 10.0 ** rng.uniform(-6, 6), 10.0 ** rng.uniform(-6, 6)
        a, b, c = _df(rng, sa), _df(rng, sb), _df(rng, sa * sb)
        if i % 5 == 0:
            b = (np.float32(-float(a[0]) * (1 + rng.uniform(-1e-6, 1e-6))), np.float32(0.0))
        ops.append((a, b, c))
    text = "\n".join(" ".join([x.hex()] + [float(v).hex() for p in o for v in p]) for x, o in zip(xs, ops)) + "\n"
    out = subprocess.run([driver], input=text, capture_output=True, text=True, check=True).stdout.split("\n")
    u2 = Fraction(1, 2**48)
    for x, (a, b, c), line in zip(xs, ops, out):
        r = [float.fromhex(t) for t in line.split()]
        hi, lo, joined = r[:3]
        if not math.isfinite(x):
            assert (math.isnan(hi) and math.isnan(x)) or hi == x
        elif x == 0.0 or abs(x) < 2.0**-126:
            assert abs(hi + lo - x) <= 2.0**-149
        elif abs(x) <= 3.4028234663852886e38:
            assert abs(Fraction(hi) + Fraction(lo) - Fraction(x)) <= u2 * abs(Fraction(x)), x
            assert joined == hi + lo
        A, B, C = _exact(*a), _exact(*b), _exact(*c)
        for got, exact, bound in ((r[3:5], A + B, 6 * u2 * (abs(A) + abs(B))),
                                  (r[5:7], A - B, 6 * u2 * (abs(A) + abs(B))),
                                  (r[7:9], A * B + C, 10 * u2 * (abs(A * B) + abs(C)))):
            assert abs(_exact(*got) - exact) <= bound
