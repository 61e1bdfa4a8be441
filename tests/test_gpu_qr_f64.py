"""The float64 QR's register form over its shapes: rows per lane and warps per column at the edges of
each, odd l, more columns than four a CTA, m = 1; columns 2^300 apart and a singular S^* (which it
leaves to the persistent kernel), tied columns, and norms that cancel all at once."""
import numpy as np
import pytest

import workloads
from tests.gpu_common import EPS, rt_module, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


def _check(torch, rt, A, l, seed):
    """R^* R = (S^* Pi)^* (S^* Pi) to 32 l eps of the larger of the two columns' norms, and every
    diagonal entry dominates its row's trailing columns."""
    m = A.shape[0]
    with rt.Projector(to_dev(torch, A), l_max=l, k_max=1, mode="fp64", rank_tol=1e-300) as P:
        S = P.sketch(seed=seed, l=l).cpu().numpy()
        P.precondition(seed=seed, l=l)
        R, perm, _ = P.export_state()
    assert sorted(perm) == list(range(m))
    assert np.all(np.tril(R, -1) == 0)
    Sp = S[perm]
    G = Sp @ Sp.T
    d = np.sqrt(np.diag(G))
    assert np.all(np.abs(R.T @ R - G) <= 32 * l * EPS * np.outer(d, d))
    tail = np.cumsum((R ** 2)[::-1], axis=0)[::-1]
    for j in range(m - 1):
        assert R[j, j] ** 2 >= (1 - 1e-9) * np.max(tail[j, j + 1:])
    return S, R, perm


@pytest.mark.parametrize("m,l", [(1, 1), (1, 7), (2, 3), (3, 383), (5, 384), (6, 385), (33, 767), (34, 769), (127, 1152),
                                 (129, 1153), (90, 1537), (60, 2304), (61, 2305), (609, 640), (700, 701), (1030, 1031)])
def test_register_qr_shapes(m, l):
    torch, rt = torch_cuda(), rt_module()
    n = max(2 * l, 64)
    _check(torch, rt, workloads.haar_spectrum_matrix(m, n, 1e-4 if m > 1 else 1.0, 300 + m + l), l, 7)


def test_columns_far_apart():
    torch, rt = torch_cuda(), rt_module()
    A = np.random.default_rng(1).standard_normal((20, 400)) * 2.0 ** -np.linspace(0, 300, 20).round()[:, None]
    S, R, perm = _check(torch, rt, A, 60, 3)
    assert list(perm[:3]) == [0, 1, 2]


def test_norms_that_cancel_at_once():
    torch, rt = torch_cuda(), rt_module()
    rng = np.random.default_rng(5)
    strong = rng.standard_normal(2048)
    A = (1.0 + 0.5 * rng.random((48, 1))) * strong[None, :] + 2.0 ** -14 * rng.standard_normal((48, 2048))
    _check(torch, rt, A, 96, 9)


def test_singular_sketch_is_reported():
    """A zero row and a repeated one: the rank check, not a wait or a wrong factor."""
    torch, rt = torch_cuda(), rt_module()
    A = np.random.default_rng(2).standard_normal((12, 300))
    A[7] = 0.0
    with rt.Projector(to_dev(torch, A), l_max=40, k_max=1, mode="fp64") as P:
        with pytest.raises(rt.RtprojError):
            P.precondition(seed=1, l=40)
