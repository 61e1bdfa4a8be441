"""The sparse form's product with A^* where a column has more entries than one 128-bit sum holds."""
import numpy as np
import pytest

from oracle import exact
from tests.gpu_common import EPS, assert_rows_close, rt_module, to_dev, torch_cuda
from tests.test_gpu_sparse_products import _irregular

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,r,heavy", [(1, 0, 2046), (1, 0, 12000), (3, 5, 20000), (20, 0, 8192), (33, 0, 9000), (70, 10, 20000)])
def test_columns_longer_than_one_sum(k, r, heavy):
    """A column of thousands of entries (duplicates, which sum), over the group widths and right-hand
    sides a lane: the tolerances of the products' tests."""
    torch, rt = torch_cuda(), rt_module()
    m, n = 48, 3001
    rp, ci, v, A = _irregular(m, n, 400 + k, heavy=heavy)
    U = V = None
    if r:
        rng = np.random.default_rng(500 + k)
        U, V = rng.standard_normal((m, r)) / np.sqrt(m * n), rng.standard_normal((r, n))
        A = A + U @ V
    B = np.random.default_rng(600 + k).standard_normal((k, n))
    Zx, ROWx, _ = exact.exact_project(A, B)
    kap = np.linalg.cond(A)
    with rt.SparseProjector(to_dev(torch, rp), to_dev(torch, ci), to_dev(torch, v), n,
                            U=None if U is None else to_dev(torch, U), V=None if V is None else to_dev(torch, V),
                            l_max=2 * m, k_max=k, refine_passes=3) as P:
        P.precondition(seed=5, l=2 * m)
        Z, ROW, _ = P.project(to_dev(torch, B), null=True, row=True)
    tol = 64 * EPS * (max(kap, 1e3) if r else 1)
    assert_rows_close(Z.cpu().numpy(), Zx, tol, "Z")
    assert_rows_close(ROW.cpu().numpy(), ROWx, 64 * tol, "ROW")
