"""The sparse form's products with zeros among large entries: right-hand sides far below them, in the
null space already, come back as they are."""
import numpy as np
import pytest

from tests.gpu_common import rt_module, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 3, 40])
def test_small_vectors_and_large_entries(k):
    """Rows (1e140, 1e140) over pairs of columns, b = (t, -t) on each pair with t down to 1e-250: A b = 0
    and h = 0 exactly, so Z = b to the bit (the products with h's zeros add nothing)."""
    torch, rt = torch_cuda(), rt_module()
    m = 12
    n = 2 * m + 3
    rp = np.arange(m + 1, dtype=np.int64) * 2
    ci = np.arange(2 * m, dtype=np.int32)
    v = np.full(2 * m, 1e140)
    B = np.zeros((k, n))
    t = 10.0 ** -np.linspace(0, 250, k * m).reshape(k, m) if k > 1 else np.full((1, m), 3.7e-230)
    B[:, 0:2 * m:2], B[:, 1:2 * m:2] = t, -t
    with rt.SparseProjector(to_dev(torch, rp), to_dev(torch, ci), to_dev(torch, v), n, l_max=n, k_max=k) as P:
        P.precondition(seed=1, l=n)
        Z, ROW, H = P.project(to_dev(torch, B), null=True, row=True, lstsq=True)
    assert np.array_equal(Z.cpu().numpy(), B)
    assert not ROW.any() and not H.any()
