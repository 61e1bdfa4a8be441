"""The float-float QR's register form over its shapes: rows per lane and warps per column at the
edges of each (l at and just past 64 rows per lane and warp), odd l, columns that do not divide
among the CTAs, more columns than four a CTA, m = 1; and a matrix whose trailing norms all
cancel at once, where the pivots are chosen again with fresh norms."""
import numpy as np
import pytest

import workloads
from tests.gpu_common import rt_module, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


def _check(torch, rt, A, l, seed):
    """Properties that do not depend on how near-ties resolve, with the bounds of the other
    float-float QR tests: R^* R = (S^* Pi)^* (S^* Pi) to 32 l 2^-48, and every diagonal entry
    dominates its row's trailing columns."""
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


@pytest.mark.parametrize("m,l", [(1, 1), (1, 7), (2, 3), (3, 191), (5, 192), (6, 193), (33, 383), (34, 385), (127, 576),
                                 (129, 577), (150, 768), (151, 769), (200, 1153), (90, 1537), (60, 2112), (61, 2305),
                                 (609, 640), (700, 701), (1030, 1031)])
def test_register_qr_shapes(m, l):
    torch, rt = torch_cuda(), rt_module()
    n = max(2 * l, 64)
    _check(torch, rt, workloads.haar_spectrum_matrix(m, n, 1e-4 if m > 1 else 1.0, 300 + m + l), l, 7)


def test_pivots_are_chosen_again_when_norms_cancel():
    """Columns of S^* that are one strong direction plus 2^-14 of their own: after the first pivot
    every trailing squared norm falls by 2^-28, far past the 2^-10 at which the early norms are
    not relied on."""
    torch, rt = torch_cuda(), rt_module()
    m, n, l = 48, 2048, 96
    rng = np.random.default_rng(5)
    strong = rng.standard_normal(n)
    A = (1.0 + 0.5 * rng.random((m, 1))) * strong[None, :] + 2.0 ** -14 * rng.standard_normal((m, n))
    _check(torch, rt, A, l, 9)
