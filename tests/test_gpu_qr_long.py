"""The register QR for columns longer than registers hold: the edges of what lies in registers, shared
memory and L2, one, two and four warps a column, odd l, one column, and the range check's fallback."""
import numpy as np
import pytest

import workloads
from tests.gpu_common import rt_module, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


def _check(torch, rt, A, l, seed):
    """R^* R = (S^* Pi)^* (S^* Pi) to 32 l 2^-48, and every diagonal entry dominates its row's trailing
    columns (the bounds of the other float-float QR tests)."""
    m = A.shape[0]
    with rt.Projector(to_dev(torch, A), l_max=l, k_max=1, rank_tol=1e-300) as P:
        S = P.sketch(seed=seed, l=l).cpu().numpy()
        P.precondition(seed=seed, l=l)
        R, perm, _ = P.export_state()
    assert sorted(perm) == list(range(m))
    assert np.all(np.tril(R, -1) == 0)
    Sp = S[perm]
    G = Sp @ Sp.T
    assert np.max(np.abs(R.T @ R - G)) <= 32 * l * 2.0 ** -48 * np.max(np.abs(G))
    tail = np.cumsum((R ** 2)[::-1], axis=0)[::-1]
    for j in range(m - 1):
        assert R[j, j] ** 2 >= (1 - 1e-6) * np.max(tail[j, j + 1:])


@pytest.mark.parametrize("m,l", [(1, 2306), (2, 4129), (5, 7000), (150, 2305), (154, 1793), (620, 1537), (700, 2801),
                                 (1217, 1218), (1217, 2049), (1400, 1600), (300, 6001), (913, 1729),
                                 (913, 1921), (913, 1728), (1060, 2112), (1060, 2113)])
def test_long_columns(m, l):
    torch, rt = torch_cuda(), rt_module()
    n = max(l, 64)
    _check(torch, rt, workloads.haar_spectrum_matrix(m, n, 1e-4 if m > 1 else 1.0, 500 + m + l), l, 7)


def test_graded_rows_fall_back():
    """Rows 2^60 apart: the float64 kernel behind takes over, and the result is the same QR."""
    torch, rt = torch_cuda(), rt_module()
    A = np.random.default_rng(3).standard_normal((40, 3000)) * 2.0 ** -np.linspace(0, 60, 40).round()[:, None]
    _check(torch, rt, A, 2500, 5)
