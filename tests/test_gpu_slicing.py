"""Digit slicing of right-hand sides: the same digits whatever the element type, the stride, the
alignment and the number of CTAs per row, and rows at the ends of the exponent range."""
import numpy as np
import pytest

import workloads
from tests.gpu_common import rt_module, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


def _matrix(m, n, seed):
    return workloads.haar_spectrum_matrix(m, n, 0.25, seed).astype(np.float32)


def _block(k, n, seed):
    B = np.random.default_rng(seed).standard_normal((k, n)).astype(np.float32)
    B *= (2.0 ** np.random.default_rng(seed + 1).integers(-30, 30, (k, 1))).astype(np.float32)
    if k > 2:
        B[1] = 0
        B[2] *= np.float32(2.0 ** -100)
        B[2, ::3] = np.float32(2.0 ** -140)             # subnormal float32 entries
    return B


@pytest.mark.parametrize("m,n,k,slices", [(5, 64, 1, 7), (20, 1001, 3, 7), (20, 1001, 3, 9), (33, 4099, 9, 7),
                                          (8, 40003, 5, 10), (40, 16384, 310, 7)])
def test_element_type_stride_and_alignment(m, n, k, slices):
    """float32 right-hand sides give what the same values in float64 give, rounded to float32;
    rows at an odd stride and offset what contiguous rows give. Bit for bit: the digits are equal."""
    torch, rt = torch_cuda(), rt_module()
    A, B = _matrix(m, n, 3), _block(k, n, m + n)
    with rt.Projector(to_dev(torch, A.astype(np.float64)), l_max=m + 4, k_max=k, apply_slices=slices) as P:
        P.precondition(seed=2, l=m + 4)
        want = P.null_project(to_dev(torch, B.astype(np.float64)))
        room = torch.zeros(k, n + 3, dtype=torch.float64, device="cuda")
        room[:, 1:n + 1] = to_dev(torch, B.astype(np.float64))
        odd = P.null_project(room[:, 1:n + 1])
    assert torch.equal(want, odd)
    with rt.Projector(to_dev(torch, A), l_max=m + 4, k_max=k, apply_slices=slices) as P:
        P.precondition(seed=2, l=m + 4)
        got = P.null_project(to_dev(torch, B))
    assert torch.equal(got, want.float())


@pytest.mark.parametrize("m,n,k", [(16, 500, 2), (16, 9000, 40)])
def test_rows_far_from_one(m, n, k):
    """Scaling a right-hand side by a power of two scales its projection exactly, at either end of
    the normal range."""
    torch, rt = torch_cuda(), rt_module()
    A = _matrix(m, n, 4).astype(np.float64)
    B = to_dev(torch, np.random.default_rng(1).standard_normal((k, n)))
    with rt.Projector(to_dev(torch, A), l_max=m + 4, k_max=k) as P:
        P.precondition(seed=2, l=m + 4)
        want = P.null_project(B)
        for e in (-850, 400):
            assert torch.equal(P.null_project(B * 2.0 ** e), want * 2.0 ** e)


def test_subnormal_rows():
    """Right-hand sides whose entries are all subnormal: c, h and Z are rounded to multiples of
    2^-1074, so with kappa = 4 and an orthonormal-scale A the result is within a few units per
    row of the projection of the integers behind them."""
    torch, rt = torch_cuda(), rt_module()
    m, n, k = 16, 700, 3
    A = _matrix(m, n, 5).astype(np.float64)
    N = np.rint(np.random.default_rng(2).standard_normal((k, n)) * 2.0 ** 30)
    with rt.Projector(to_dev(torch, A), l_max=m + 4, k_max=k) as P:
        P.precondition(seed=2, l=m + 4)
        want = P.null_project(to_dev(torch, N)).cpu().numpy()
        got = P.null_project(to_dev(torch, N * 2.0 ** -1074)).cpu().numpy()
    assert np.max(np.abs(got * 2.0 ** 1000 * 2.0 ** 74 - want)) <= 64 * m
