"""The sparse form's launch shapes: the sketch by one or several panels a launch, the Gram's columns by 4
to 32 a turn, A x with narrow and wide groups of lanes."""
import numpy as np
import pytest

import tests.test_gpu_sparse_gram as gram
import tests.test_gpu_sparse_sketch as sketch
from oracle import exact
from tests.gpu_common import EPS, assert_rows_close, rt_module, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,l,r,dist", [(7, 500, 130, 2, "gaussian"), (15, 900, 65, 0, "uniform"), (16, 700, 200, 0, "gaussian"),
                                          (33, 900, 260, 13, "gaussian"), (33, 900, 128, 0, "rademacher"), (130, 1500, 520, 64, "uniform"),
                                          (64, 60001, 300, 3, "gaussian"), (40, 90001, 161, 0, "gaussian")])
def test_sketch_of_several_panels(m, n, l, r, dist):
    """Storage for one panel only (m < 16, or 16 to 31 rows), for some of them, for all; more than stay in
    L2 together: the sketch test's bound."""
    sketch.test_sketch_matches_a_dense_product(m, n, l, r, dist, 0)


@pytest.mark.parametrize("m,n,r", [(3, 5, 0), (4, 6, 2), (20, 12161, 3), (20, 40001, 0), (20, 40001, 3), (300, 19500, 2)])
def test_gram_by_columns_a_turn(m, n, r):
    gram.test_gram_matches_the_definition(m, n, r, 0)


@pytest.mark.parametrize("m,n,k,r", [(3, 900, 129, 0), (30, 900, 5, 2), (650, 1400, 1, 0), (650, 1400, 17, 0), (650, 1400, 33, 3),
                                     (320, 1400, 40, 0), (5, 40001, 17, 0)])
def test_products_by_groups_of_lanes(m, n, k, r):
    """Few chunks of nonzeros (narrow groups share a chunk) and enough of them for whole warps: the
    tolerances of the products' tests."""
    torch, rt = torch_cuda(), rt_module()
    rng = np.random.default_rng(m + n + k)
    per = rng.integers(1, 6, n)
    col = np.repeat(np.arange(n), per).astype(np.int32)
    row = rng.integers(0, m, col.size)
    row[np.cumsum(per) - per] = np.arange(n) % m
    val = np.round(rng.standard_normal(col.size) * 2.0 ** 20) / 2.0 ** 20       # sums of duplicates stay exact
    order = np.argsort(row, kind="stable")
    row, col, val = row[order], col[order], val[order]
    rp = np.concatenate([[0], np.cumsum(np.bincount(row, minlength=m))]).astype(np.int64)
    A = np.zeros((m, n))
    np.add.at(A, (row, col), val)
    U = V = None
    if r:
        U, V = rng.standard_normal((m, r)) / np.sqrt(m * n), rng.standard_normal((r, n))
        A = A + U @ V
    B = rng.standard_normal((k, n))
    few = min(k, 4)
    Zx, ROWx, _ = exact.exact_project(A, B[:few])
    with rt.SparseProjector(to_dev(torch, rp), to_dev(torch, col), to_dev(torch, val), n,
                            U=None if U is None else to_dev(torch, U), V=None if V is None else to_dev(torch, V),
                            l_max=m + 4 if m > 40 else 2 * m, k_max=k, refine_passes=3) as P:
        P.precondition(seed=5)
        Z, ROW, H = P.project(to_dev(torch, B), null=True, row=True, lstsq=True)
        back = P.project(to_dev(torch, B[::-1].copy()), null=True)[0].flip(0)
    tol = 64 * EPS * (max(np.linalg.cond(A), 1e3) if r else 1)
    assert_rows_close(Z.cpu().numpy()[:few], Zx, tol, "Z")
    assert_rows_close(ROW.cpu().numpy()[:few], ROWx, 64 * tol, "ROW")
    assert_rows_close(back.cpu().numpy(), Z.cpu().numpy(), 2 * tol, "the vectors in the other order")


@pytest.mark.parametrize("r,spike", [(0, False), (1, False), (5, False), (5, True), (20, True)])
@pytest.mark.parametrize("m,n", [(20, 23), (33, 150), (300, 700), (25, 9000)])
def test_gram_with_long_columns(m, n, r, spike):
    """Columns of some hundreds to thousands of entries (duplicates that sum), which go one a turn where
    columns are few; V by limbs or, with one large entry a row, in float64. L L^* against W W^*,
    W = R^{-*} Pi A: the Gram test's bound with its terms counted as the longest column's."""
    torch, rt = torch_cuda(), rt_module()
    rng = np.random.default_rng(m + n + r)
    per = rng.integers(1, 6, n)
    longest = 1500
    cols = rng.choice(n, 3, replace=False)
    col = np.concatenate([np.repeat(np.arange(n), per), np.full(longest, cols[0]), np.full(300, cols[1]), np.full(257, cols[2])])
    row = rng.integers(0, m, col.size)
    row[np.cumsum(per) - per] = np.arange(n) % m
    val = rng.standard_normal(col.size)
    val[per.sum():] *= 0.05
    order = np.argsort(row, kind="stable")
    row, col, val = row[order], col[order].astype(np.int32), val[order]
    rp = np.concatenate([[0], np.cumsum(np.bincount(row, minlength=m))]).astype(np.int64)
    A = np.zeros((m, n))
    np.add.at(A, (row, col), val)
    U = V = None
    if r:
        r = min(r, m)
        U, V = rng.standard_normal((m, r)) / np.sqrt(r) / 8, rng.standard_normal((r, n))
        if spike:
            V[np.arange(r), rng.integers(0, n, r)] *= 64.0
        A = A + U @ V
    kappa = np.linalg.cond(A)
    assert kappa < 1e4
    l = min(n, 2 * m + 8)
    with rt.SparseProjector(to_dev(torch, rp), to_dev(torch, col), to_dev(torch, val), n,
                            U=None if U is None else to_dev(torch, U), V=None if V is None else to_dev(torch, V),
                            l_max=l) as P:
        P.precondition(seed=3, l=l)
        R, perm, L = P.export_state()
    W = np.linalg.solve(R.T, A[perm])
    X = W @ W.T
    L = np.tril(L)
    assert np.max(np.abs(L @ L.T - X)) <= 2 * longest * kappa ** 2 * 2.0 ** -50 * np.max(np.abs(X))
