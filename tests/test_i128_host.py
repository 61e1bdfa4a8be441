"""The 128-bit sums of exact products behind the sparse form's apply (csrc/i128.cuh),
compiled for the host from the same source and checked with exact rationals: a sum of N
products is within N 2^-105 of its largest product (the bound the kernels rely on), the
rounded result is the nearest double of a value within that bound, and the pair form holds
it to 106 bits. Signs, exponents 600 apart, subnormals, zeros and full chunks of 2048."""
import os
import shutil
import subprocess
from fractions import Fraction as F

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def i128(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path_factory.mktemp("i128") / "i128")
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-w", "-I",
                    os.path.join(ROOT, "paper_0912_1135_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "i128_host_check.cpp"), "-o", exe], check=True)

    def run(op, xs, ys):
        text = f"{op} {len(xs)}\n" + "\n".join(f"{x.hex()} {y.hex()}" for x, y in zip(xs, ys)) + "\n"
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True)
        return [float.fromhex(v) for v in out.stdout.split()]
    return run


def _draw(kind, n, seed):
    rng = np.random.default_rng(seed)
    x, y = rng.standard_normal(n), rng.standard_normal(n)
    if kind == "wide":                     # exponents far apart, growing and shrinking
        x = x * 2.0 ** rng.integers(-300, 300, n)
        y = y * 2.0 ** rng.integers(-300, 300, n)
    elif kind == "cancel":                 # pairs that cancel but for their last bits
        x[1::2] = -x[::2][: len(x[1::2])] * (1 + 2.0 ** -50)
        y[1::2] = y[::2][: len(y[1::2])]
    elif kind == "full":                   # every product at the top of its binade, one sign
        x, y = np.full(n, 2.0 - 2.0 ** -52), np.full(n, 2.0 - 2.0 ** -52)
        y[2::3] *= -1                      # the check flips the sign of every third product
    elif kind == "tiny":                   # subnormals and zeros
        x = x * 2.0 ** -1040
        x[::4] = 0.0
    return [float(v) for v in x], [float(v) for v in y]


@pytest.mark.parametrize("op", ["sum", "two"])
@pytest.mark.parametrize("kind,n", [("plain", 1), ("plain", 37), ("plain", 2048), ("wide", 200), ("cancel", 64),
                                    ("full", 2048), ("tiny", 50)])
def test_sum_of_products(i128, op, kind, n):
    for seed in range(4):
        xs, ys = _draw(kind, n, seed)
        prods = [F(x) * F(y) * (-1 if i % 3 == 2 else 1) for i, (x, y) in enumerate(zip(xs, ys))]
        exact, top = sum(prods), max(abs(p) for p in prods)
        got, hi, lo = i128(op, xs, ys)
        bound = (n + 1) * top / 2 ** 105
        assert abs(F(hi) + F(lo) - exact) <= bound + abs(exact) / 2 ** 105 + F(1, 2 ** 1074)
        assert abs(F(got) - exact) <= bound + abs(exact) / 2 ** 53 + F(1, 2 ** 1074)
        assert abs(lo) <= abs(hi) * 2.0 ** -51 or hi == 0.0
