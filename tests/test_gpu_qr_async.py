"""The pivoted QRs of asynchronous handles: the persistent float-float kernel (columns in shared memory,
or in global memory where they do not fit), the persistent float64 kernel (both), and the register form
for up to 100 columns."""
import numpy as np
import pytest

import workloads
from tests.gpu_common import EPS, rt_module, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,m,l", [("mixed", 100, 104), ("mixed", 101, 104), ("mixed", 333, 698), ("mixed", 512, 516),
                                      ("mixed", 609, 1500), ("mixed", 700, 5000), ("mixed", 1030, 4128),
                                      ("fp64", 60, 64), ("fp64", 256, 544), ("fp64", 609, 700), ("fp64", 700, 5001)])
def test_pivoted_qr_of_an_asynchronous_handle(mode, m, l):
    """R^* R = (S^* Pi)^* (S^* Pi) to 32 l units of the arithmetic (2^-48 or eps), R upper triangular, and
    every diagonal entry dominates its row's trailing columns: the bounds of the other QR tests."""
    torch, rt = torch_cuda(), rt_module()
    A = workloads.haar_spectrum_matrix(m, l, 1e-4, 700 + m + l)
    with rt.Projector(to_dev(torch, A), l_max=l, k_max=1, mode=mode, rank_tol=1e-300, async_=1) as P:
        S = P.sketch(seed=9, l=l).cpu().numpy()
        P.precondition(seed=9, l=l)
        R, perm, _ = P.export_state()
        assert P.info()["status"] == 0
    assert sorted(perm) == list(range(m))
    assert np.all(np.tril(R, -1) == 0)
    Sp = S[perm]
    G = Sp @ Sp.T
    unit = EPS if mode == "fp64" else 2.0 ** -48
    assert np.max(np.abs(R.T @ R - G)) <= 32 * l * unit * np.max(np.abs(G))
    tail = np.cumsum((R ** 2)[::-1], axis=0)[::-1]
    for j in range(m - 1):
        assert R[j, j] ** 2 >= (1 - 1e-6) * np.max(tail[j, j + 1:])
