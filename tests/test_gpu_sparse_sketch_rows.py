"""The sparse sketch by lengths of rows: short ones, for which G is generated in place, long ones shared by
several CTAs, of one chunk of nonzeros or more each, with several panels a launch."""
import numpy as np
import pytest

import tests.test_gpu_sparse_sketch as sketch
from tests.gpu_common import EPS, rt_module, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dist", ["gaussian", "uniform", "rademacher"])
@pytest.mark.parametrize("m,n,l", [(1, 1, 1), (5, 30, 7), (40, 300, 64), (40, 300, 65), (70, 301, 200)])
@pytest.mark.parametrize("longest", [16, 17])
def test_short_rows(m, n, l, dist, longest):
    """Rows of up to 16 nonzeros (17: by panels), each entry within 64 eps sum |A||G|."""
    torch, rt = torch_cuda(), rt_module()
    rng = np.random.default_rng(m + n + l)
    cnt = rng.integers(0, min(n, 16) + 1, m)
    cnt[0] = min(n, longest)
    rp = np.concatenate([[0], np.cumsum(cnt)]).astype(np.int64)
    ci = np.concatenate([np.sort(rng.choice(n, c, replace=False)) for c in cnt]).astype(np.int32)
    v = rng.standard_normal(ci.size)
    A = np.zeros((m, n))
    A[np.repeat(np.arange(m), cnt), ci] = v
    with rt.SparseProjector(to_dev(torch, rp), to_dev(torch, ci), to_dev(torch, v), n, l_max=l, omega=dist) as P:
        S = P.sketch(11, l).cpu().numpy()
    G = rt.generate_omega(11, n, l, dist).cpu().numpy()
    assert np.all(np.abs(S - A @ G) <= 64 * EPS * (np.abs(A) @ np.abs(G)))


@pytest.mark.parametrize("m,n,l,r,dist", [(1, 900, 5, 0, "gaussian"), (2, 3000, 200, 1, "uniform"), (20, 30001, 150, 0, "gaussian"),
                                          (33, 20000, 260, 13, "rademacher"), (3, 620001, 5, 0, "gaussian")])
def test_long_rows(m, n, l, r, dist):
    """Rows of many chunks (the first has a good part of all nonzeros): the sketch test's bound."""
    sketch.test_sketch_matches_a_dense_product(m, n, l, r, dist, 0)
