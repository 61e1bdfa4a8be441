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
        if op == "sub":
            text = f"sub {len(xs)}\n" + "\n".join(
                f"{x.hex()} " + " ".join("%x" % ((v >> (32 * i)) & 0xFFFFFFFF) for i in range(4)) + f" {e}"
                for x, (v, e) in zip(xs, ys)) + "\n"
            out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True)
            return [(int(a), float.fromhex(b), float.fromhex(c)) for a, b, c in map(str.split, out.stdout.splitlines())]
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


@pytest.mark.parametrize("kind,n", [("plain", 2047), ("plain", 2048), ("plain", 2049), ("plain", 4160), ("full", 4160),
                                    ("wide", 4160), ("cancel", 10000), ("plain", 50000), ("full", 50000)])
def test_sum_of_any_length(i128, kind, n):
    """Sums longer than one integer holds, in P parts: each part's terms and its pair lose 2^-105 of the
    largest product (of the part) a term, and each of the P additions in double-double at most 2^-103
    of the two magnitudes added, N times the largest product each."""
    for seed in range(2):
        xs, ys = _draw(kind, n, 50 + seed)
        prods = [F(x) * F(y) * (-1 if i % 3 == 2 else 1) for i, (x, y) in enumerate(zip(xs, ys))]
        exact, top = sum(prods), max(abs(p) for p in prods)
        got, hi, lo = i128("long", xs, ys)
        bound = (2 + 8 * (n // 2048 + 1)) * (n + 1) * top / 2 ** 105
        assert abs(F(hi) + F(lo) - exact) <= bound
        assert abs(F(got) - exact) <= bound + abs(exact) / 2 ** 53


def test_rounding_and_difference(i128):
    """V 2^e is rounded to the nearest double, ties to even, and x - V 2^e is the exact
    difference rounded once wherever the two units lie close enough for it to be taken (always
    when x's last place is within 22 bits below and 63 above V's unit)."""
    rng = np.random.default_rng(9)
    xs, vs = [], []
    for i in range(4000):
        bits = int(rng.integers(1, 104))
        v = int.from_bytes(rng.bytes(16), "little") >> (128 - bits)
        if i % 5 == 0 and bits > 54:                     # exact ties and their neighbours
            v = (v >> (bits - 53) << (bits - 53)) + (1 << (bits - 54)) + int(rng.integers(-1, 2))
        v = -v if rng.random() < 0.5 else v
        e = int(rng.integers(-200, 100))
        x = float(rng.standard_normal()) * 2.0 ** (e + int(rng.integers(-30, 130)))
        if i % 7 == 0:
            x = float(F(v) * F(2) ** e) * (1 + 2.0 ** -52 * int(rng.integers(-2, 3)))   # cancels
        xs.append(x if i % 11 else 0.0)
        vs.append((v, e))
    taken = 0
    for x, (v, e), (ok, diff, val) in zip(xs, vs, i128("sub", xs, vs)):
        exact = F(v) * F(2) ** e
        assert val == float(exact)                       # Fraction to float rounds to nearest even
        m, ex = np.frexp(x)
        place = int(ex) - 53 - e                         # x's last place above V's unit
        if x != 0.0:
            assert bool(ok) == (-22 <= place <= 63)
        if ok:
            taken += 1
            assert diff == float(F(x) - exact)
    assert taken > 1000
