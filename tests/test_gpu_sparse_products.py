"""The sparse form's products with A and A^* over every layout of right-hand sides: one lane
group of 1, 2, 4, ..., 32 lanes and one to four right-hand sides a lane, with and without a
low-rank term, rows longer than one chunk, a column with more entries than one sum holds, and
an infinity among the right-hand sides."""
import numpy as np
import pytest

from oracle import exact
from tests.gpu_common import EPS, assert_rows_close, rt_module, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


def _irregular(m, n, seed, heavy=0):
    """Two to six entries a column in random rows (row 0 gets most), rows of different scales;
    `heavy` extra entries (duplicates that sum) in column 3."""
    rng = np.random.default_rng(seed)
    per = rng.integers(2, 7, n)
    col = np.repeat(np.arange(n), per)
    row = np.minimum((m * rng.random(col.size) ** 3).astype(int), m - 1)
    row[np.cumsum(per) - per] = np.arange(n) % m
    val = rng.standard_normal(col.size)
    if heavy:
        col = np.concatenate([col, np.full(heavy, 3)])
        row = np.concatenate([row, rng.integers(0, m, heavy)])
        val = np.concatenate([val, rng.integers(-8, 9, heavy) / 64.0])
    val = np.round(val * 2.0 ** 20) / 2.0 ** 20 * 2.0 ** (-(row % 11))    # sums of duplicates stay exact
    order = np.argsort(row, kind="stable")
    row, col, val = row[order], col[order], val[order]
    rp = np.concatenate([[0], np.cumsum(np.bincount(row, minlength=m))]).astype(np.int64)
    A = np.zeros((m, n))
    np.add.at(A, (row, col), val)
    return rp, col.astype(np.int32), val, A


@pytest.mark.parametrize("k,r", [(1, 0), (1, 3), (2, 0), (3, 10), (7, 0), (16, 0), (17, 5), (33, 0), (70, 10), (129, 0)])
def test_every_group_width_matches_the_exact_projection(k, r):
    """Z and the row-space projection within 64 eps of the exact projection (the tolerance of the
    sparse form's closed-form tests; with a low-rank term the dense sum is rounded once, so times
    its condition number floored at 1e3), and h within 64 eps kappa."""
    torch, rt = torch_cuda(), rt_module()
    m, n = 48, 9001
    rp, ci, v, A = _irregular(m, n, 100 + k, heavy=3000 if k == 7 else 0)
    U = V = None
    if r:
        rng = np.random.default_rng(200 + k)
        U, V = rng.standard_normal((m, r)) / np.sqrt(m * n), rng.standard_normal((r, n))
        A = A + U @ V
    B = np.random.default_rng(300 + k).standard_normal((k, n))
    Zx, ROWx, Hx = exact.exact_project(A, B)
    kap = np.linalg.cond(A)
    with rt.SparseProjector(to_dev(torch, rp), to_dev(torch, ci), to_dev(torch, v), n,
                            U=None if U is None else to_dev(torch, U), V=None if V is None else to_dev(torch, V),
                            l_max=2 * m, k_max=k, refine_passes=3) as P:
        P.precondition(seed=5, l=2 * m)
        Z, ROW, H = P.project(to_dev(torch, B), null=True, row=True, lstsq=True)
        out = to_dev(torch, B)
        P.null_project(out, out=out)                    # in place
        assert torch.equal(out, Z)
        bad = to_dev(torch, B)
        bad[k // 2, 11] = float("inf")
        Zb = P.null_project(bad)
        assert not torch.isfinite(Zb[k // 2]).all()
        if k > 1:                                       # the other vectors are untouched by it
            keep = [j for j in range(k) if j != k // 2]
            assert torch.equal(Zb[keep], Z[keep])
    tol = 64 * EPS * (max(kap, 1e3) if r else 1)
    assert_rows_close(Z.cpu().numpy(), Zx, tol, "Z")
    assert_rows_close(ROW.cpu().numpy(), ROWx, 64 * tol, "ROW")
    H = H.cpu().numpy()
    assert np.max(np.linalg.norm(H - Hx, axis=1) / np.linalg.norm(Hx, axis=1)) <= 64 * EPS * max(kap, 1e3)
