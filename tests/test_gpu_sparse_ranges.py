"""The sparse form's low-rank factors over their range: rows of V that span 2^40 and more (one huge entry,
columns scaled apart, half of the rows small in half of the columns), a row of zeros, a row of
subnormals. The preconditioner is as good as float64 allows, and Z is the exact projection."""
import numpy as np
import pytest

from oracle import exact
from tests.gpu_common import EPS, assert_rows_close, rt_module, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


def _matrix(m, n, seed, dense=True):
    rng = np.random.default_rng(seed)
    per = rng.integers(2, 7, n)
    col = np.repeat(np.arange(n), per).astype(np.int32)
    row = rng.integers(0, m, col.size)
    row[np.cumsum(per) - per] = np.arange(n) % m
    val = rng.standard_normal(col.size)
    order = np.argsort(row, kind="stable")
    row, col, val = row[order], col[order], val[order]
    S = np.zeros((m, n)) if dense else None
    if dense:
        np.add.at(S, (row, col), val)
    return rng, np.concatenate([[0], np.cumsum(np.bincount(row, minlength=m))]).astype(np.int64), col, val, S


@pytest.mark.parametrize("kind", ["plain", "spike", "columns", "block", "zero", "subnormal"])
@pytest.mark.parametrize("m,n,r", [(40, 900, 6), (64, 5003, 10)])
def test_low_rank_factors_of_wide_range(m, n, r, kind):
    """T = L^{-1} R^{-*} Pi makes T A A^* T^* the identity up to E's rounding in float64, scaled by R^{-*}:
    m eps kappa(R). One huge entry a row of V puts 2^40
    into kappa(R) itself; the others leave it as it is. Z after three passes: 64 eps kappa(R), floored
    at 1e3 (the dense sum is rounded once)."""
    torch, rt = torch_cuda(), rt_module()
    rng, rp, ci, v, S = _matrix(m, n, m + n + len(kind))
    U, V = rng.standard_normal((m, r)) / np.sqrt(r), rng.standard_normal((r, n))
    if kind == "spike":
        V[np.arange(r), rng.permutation(n)[:r]] *= 2.0 ** 40
        U[r + 2:] = 0.0
    elif kind == "columns":
        V *= 2.0 ** (-60.0 * rng.random(n)).round()
    elif kind == "block":
        V[: r // 2, : n // 2] *= 2.0 ** -40
        U[r + 2:] = 0.0
    elif kind == "zero":
        V[r // 2] = 0.0
    elif kind == "subnormal":
        V[r // 2] *= 2.0 ** -1050
    A = S + U @ V
    with rt.SparseProjector(to_dev(torch, rp), to_dev(torch, ci), to_dev(torch, v), n, U=to_dev(torch, U), V=to_dev(torch, V),
                            l_max=2 * m, k_max=2, refine_passes=3, rank_tol=1e-300) as P:
        P.precondition(seed=4, l=2 * m)
        R, perm, L = P.export_state()
        B = rng.standard_normal((2, n))
        Z = P.null_project(to_dev(torch, B)).cpu().numpy()
    kappa_r = np.linalg.cond(R)
    W = np.linalg.solve(R.T, A[perm])                # R^{-*} Pi A
    T = np.linalg.solve(np.tril(L), W)
    assert np.linalg.norm(T @ T.T - np.eye(m), 2) <= m * EPS * max(kappa_r, 1e2)
    if kind != "spike":
        assert kappa_r < 1e3
        Zx, _, _ = exact.exact_project(A, B)
        assert_rows_close(Z, Zx, 64 * EPS * 1e3, "Z")


@pytest.mark.parametrize("kind", ["spike", "columns"])
def test_first_correction_is_float64s(kind):
    """Rows of V with one entry 2^12 times the others, or over columns 2^40 apart, and many columns: the
    first pass's ||dh|| / ||h|| is what a float64 Gram matrix leaves, eps kappa(R) and a factor of 2
    (fixed point against the rows' largest entries lost 8 of the bits)."""
    torch, rt = torch_cuda(), rt_module()
    m, n, r = 100, 200000, 10
    for seed in range(3):
        rng, rp, ci, v, _ = _matrix(m, n, seed, dense=False)
        U, V = rng.standard_normal((m, r)) / np.sqrt(r), rng.standard_normal((r, n))
        if kind == "spike":
            V[np.arange(r), rng.permutation(n)[:r]] *= 2.0 ** 12
            U[r + 2:] = 0.0
        else:
            V *= 2.0 ** (-40.0 * rng.random(n))
        with rt.SparseProjector(to_dev(torch, rp), to_dev(torch, ci), to_dev(torch, v), n, U=to_dev(torch, U),
                                V=to_dev(torch, V), l_max=m + 4, k_max=2, refine_passes=1, rank_tol=1e-300) as P:
            P.precondition(seed=3, l=m + 4)
            P.null_project(to_dev(torch, rng.standard_normal((2, n))))
            info = P.info()
        assert info["dh_rel"] <= 2 * EPS * info["kappa_R"], (seed, info["dh_rel"], info["kappa_R"])
