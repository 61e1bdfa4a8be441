"""Zero and subnormal factors in the 128-bit sums of exact products (csrc/i128.cuh): beside a huge other
factor they must not move the sum's unit past what their product is."""
from fractions import Fraction as F

import numpy as np
import pytest

from tests.test_i128_host import i128  # noqa: F401  (the fixture)


@pytest.mark.parametrize("op", ["sum", "two", "long"])
@pytest.mark.parametrize("n", [1, 60, 2048])
def test_zero_and_subnormal_factors(i128, op, n):  # noqa: F811
    """N products within (N + 1) 2^-105 of the largest (the sums' bound, a subnormal factor counted as
    2^-1022), the result rounded once."""
    size = lambda v: F(max(abs(v), 2.0 ** -1022)) if v else F(0)  # noqa: E731
    for seed in range(4):
        rng = np.random.default_rng(100 + seed)
        x, y = rng.standard_normal(n) * 2.0 ** -340, rng.standard_normal(n) * 2.0 ** -340
        x[1::3], y[1::3] = 2.0 ** 600, 0.0
        x[2::5], y[2::5] = 2.0 ** 500 * (1 + 2.0 ** -52), 2.0 ** -1074 * rng.integers(0, 4, len(y[2::5]))
        x[3::7], y[3::7] = 2.0 ** -1074 * rng.integers(0, 4, len(x[3::7])), 2.0 ** 450 * (1 - 2.0 ** -53)
        xs, ys = [float(v) for v in x], [float(v) for v in y]
        prods = [F(u) * F(v) * (-1 if i % 3 == 2 else 1) for i, (u, v) in enumerate(zip(xs, ys))]
        exact, top = sum(prods), max(size(u) * size(v) for u, v in zip(xs, ys))
        got, hi, lo = i128(op, xs, ys)
        bound = 2 * (n + 1) * top / 2 ** 105 + abs(exact) / 2 ** 105
        assert abs(F(hi) + F(lo) - exact) <= bound
        assert abs(F(got) - exact) <= bound + abs(exact) / 2 ** 53
