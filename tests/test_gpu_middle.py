"""The apply's middle h = Pi^* T1^* T1 Pi c for small m^2 k, summed from exact products: against
the sliced form on the other side of the rule, and against float64 where that side is far."""
import numpy as np
import pytest

import workloads
from tests.gpu_common import rt_module, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

PRODUCTS = 4 << 20     # the rule: m^2 k up to this many products are summed directly,
                       # k rounded up to a power of two, or to a multiple of 32
KAPPA = 4.0


def _matrix(m, seed):
    return workloads.haar_spectrum_matrix(m, 4 * m + 32, 1.0 / KAPPA if m > 1 else 1.0, seed)


@pytest.mark.parametrize("m,k", [(1, 1), (2, 3), (5, 1), (7, 40), (31, 2), (32, 16)])
def test_small_blocks_against_float64(m, k):
    """Unrefined least squares: the preconditioner's own error is that of its Gram digits, at
    least 32 bits, times kappa^2 and a sum over m: 2^-20 covers m <= 32."""
    torch, rt = torch_cuda(), rt_module()
    A = _matrix(m, 40 + m)
    B = np.random.default_rng(m + k).standard_normal((k, A.shape[1]))
    want = np.linalg.solve(A @ A.T, A @ B.T).T
    with rt.Projector(to_dev(torch, A), l_max=m + 4, k_max=k, refine_passes=0) as P:
        P.precondition(seed=5, l=m + 4)
        X = P.lstsq(to_dev(torch, B)).cpu().numpy()
    assert np.max(np.abs(X - want)) <= 2.0 ** -20 * np.max(np.abs(want))


@pytest.mark.parametrize("m,ks", [(33, (1, 3, 33)), (64, (1, 17)), (65, (32, 64)), (127, (5, 100)), (300, (1, 7, 32)),
                                  (513, (2, 5, 8)), (1023, (1, 3)), (2048, (1,))])
def test_direct_and_sliced_forms_agree(m, ks):
    """One handle, blocks on both sides of the rule. Each form takes its two products to
    m 2^-52 relative to |D||c| (D = T1 Pi, ||D||^2 = kappa^2 / ||A||^2), so the results differ by at
    most 4 m 2^-52 times m kappa^2 of the largest entry of h."""
    torch, rt = torch_cuda(), rt_module()
    big = PRODUCTS // (m * m) + 1
    assert all(m * m * (1 << (k - 1).bit_length() if k <= 32 else -(-k // 32) * 32) <= PRODUCTS for k in ks)
    A = _matrix(m, 60 + m)
    B = to_dev(torch, np.random.default_rng(m).standard_normal((big, A.shape[1])))
    with rt.Projector(to_dev(torch, A), l_max=m + 4, k_max=big, refine_passes=0) as P:
        P.precondition(seed=5, l=m + 4)
        want = P.lstsq(B).cpu().numpy()
        for k in ks:
            got = P.lstsq(B[:k].contiguous()).cpu().numpy()
            assert np.max(np.abs(got - want[:k])) <= 4 * m * 2.0 ** -52 * m * KAPPA ** 2 * np.max(np.abs(want))


def test_more_columns_than_a_grid_dimension():
    """m = 1 with k past 65535 groups of 32 columns: every row of Z is b - (a b) a^* / (a a^*)."""
    torch, rt = torch_cuda(), rt_module()
    k, n = 65535 * 32 + 33, 8
    A = np.random.default_rng(1).standard_normal((1, n))
    B = torch.randn(k, n, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    with rt.Projector(to_dev(torch, A), l_max=n, k_max=k) as P:
        P.precondition(seed=5, l=n)
        Z = P.null_project(B)
    a = to_dev(torch, A)
    want = B - (B @ a.T) @ a / (a @ a.T)
    assert float((Z - want).abs().max()) <= 64 * 2.0 ** -52 * float(B.abs().max())
