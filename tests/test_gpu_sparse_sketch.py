"""The sparse sketch by panels of G: every width of the last panel, fewer rows than the panel's
place in D needs (m < 16), rows of one nonzero and rows longer than one pass, values whose sizes
differ by 2^80 within a row, empty rows, low-rank terms up to 64, all distributions."""
import numpy as np
import pytest

from tests.gpu_common import EPS, rt_module, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,l,r,dist,spread", [(3, 40, 3, 0, "gaussian", 0), (15, 333, 64, 0, "uniform", 0),
                                                 (16, 700, 65, 1, "rademacher", 0), (40, 5000, 127, 9, "gaussian", 0),
                                                 (70, 3001, 129, 64, "uniform", 0), (24, 9000, 200, 13, "gaussian", 80),
                                                 (5, 20001, 6, 5, "rademacher", 40)])
def test_sketch_matches_a_dense_product(m, n, l, r, dist, spread):
    """Against A G with the stored G, each entry within 64 eps sum |A||G| (the bound of the sparse
    form's other sketch test) and, for values spread over many binades, 64 eps times the row's
    largest value times sum |G| over its nonzeros' columns (the documented error of the limbs
    lies far inside it)."""
    torch, rt = torch_cuda(), rt_module()
    rng = np.random.default_rng(m + n)
    per = rng.integers(1, 9, n)
    col = np.repeat(np.arange(n), per).astype(np.int32)
    row = np.minimum((m * rng.random(col.size) ** 2).astype(np.int64), m - 1)
    if m > 4:
        row[row == 1] = 0                                  # row 1 is empty
        row[0] = 2
    val = rng.standard_normal(col.size) * 2.0 ** -rng.integers(0, spread + 1, col.size)
    order = np.argsort(row, kind="stable")
    row, col, val = row[order], col[order], val[order]
    rp = np.concatenate([[0], np.cumsum(np.bincount(row, minlength=m))]).astype(np.int64)
    A = np.zeros((m, n))
    np.add.at(A, (row, col), val)
    absA, big = np.abs(A), np.zeros((m, n))
    top = np.zeros(m)
    np.maximum.at(top, row, np.abs(val))
    big[row, col] = top[row]
    U = V = None
    if r:
        U, V = rng.standard_normal((m, r)), rng.standard_normal((r, n))
        A = A + U @ V
        low = np.abs(U) @ np.abs(V)
        absA, big = absA + low, big + low
    with rt.SparseProjector(to_dev(torch, rp), to_dev(torch, col), to_dev(torch, val), n,
                            U=None if U is None else to_dev(torch, U), V=None if V is None else to_dev(torch, V),
                            l_max=l, omega=dist) as P:
        S = P.sketch(7, l).cpu().numpy()
    G = rt.generate_omega(7, n, l, dist).cpu().numpy()
    bound = 64 * EPS * ((absA if spread == 0 else big) @ np.abs(G))
    assert np.all(np.abs(S - A @ G) <= bound + 1e-300)
