"""The sparse form's Gram matrix with a low-rank term: D = A^* P^- and V D by limbs, over ranks at
the edges of the groups of V's rows and of the sums' capacity, k past one CTA's threads, ragged n,
and factors whose rows are scaled apart."""
import numpy as np
import pytest

from tests.gpu_common import rt_module, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,r,spread", [(7, 61, 1, 0), (20, 1000, 4, 0), (33, 3001, 5, 60), (40, 20011, 10, 0),
                                          (50, 4097, 12, 200), (64, 2500, 13, 0), (64, 2500, 16, 0), (70, 2500, 17, 40),
                                          (100, 5000, 33, 0), (128, 6000, 64, 100), (257, 4000, 10, 0), (600, 9000, 2, 0),
                                          (300, 5000, 0, 0)])
def test_gram_matches_the_definition(m, n, r, spread):
    """L L^* against W W^*, W = R^{-*} Pi A, in extended precision. D carries 2^-53 of the partial
    sums of |A||P^-| and the rest 2^-53 of products of norms 1 and kappa: 2 m kappa^2 2^-50 of the
    largest entry covers m terms a sum and the Cholesky factor."""
    torch, rt = torch_cuda(), rt_module()
    rng = np.random.default_rng(m + n + r)
    per = rng.integers(1, 6, n)
    col = np.repeat(np.arange(n), per).astype(np.int32)
    row = rng.integers(0, m, col.size)
    val = rng.standard_normal(col.size)
    order = np.argsort(row, kind="stable")
    row, col, val = row[order], col[order], val[order]
    rp = np.concatenate([[0], np.cumsum(np.bincount(row, minlength=m))]).astype(np.int64)
    A = np.zeros((m, n))
    np.add.at(A, (row, col), val)
    U = V = None
    if r:
        scale = 2.0 ** rng.integers(-spread, spread + 1, (r, 1))
        U, V = rng.standard_normal((m, r)) / np.sqrt(r) / scale.T, rng.standard_normal((r, n)) * scale
        A = A + U @ V
    kappa = np.linalg.cond(A)
    assert kappa < 1e3
    l = min(n, 2 * m + 8)
    with rt.SparseProjector(to_dev(torch, rp), to_dev(torch, col), to_dev(torch, val), n,
                            U=None if U is None else to_dev(torch, U), V=None if V is None else to_dev(torch, V),
                            l_max=l) as P:
        P.precondition(seed=3, l=l)
        R, perm, L = P.export_state()
    W = np.linalg.solve(R.T, A[perm])
    X = W @ W.T
    L = np.tril(L)
    assert np.max(np.abs(L @ L.T - X)) <= 2 * m * kappa ** 2 * 2.0 ** -50 * np.max(np.abs(X))
