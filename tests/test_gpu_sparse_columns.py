"""Column indices out of range beside a low-rank term: refused at create, and never used to index V."""
import numpy as np
import pytest

from tests.gpu_common import rt_module, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [-1, -2 ** 31, 400, 2 ** 31 - 1])
def test_column_index_out_of_range_with_a_low_rank_term(bad):
    torch, rt = torch_cuda(), rt_module()
    rng = np.random.default_rng(1)
    m, n, r = 10, 400, 3
    rp = np.arange(m + 1, dtype=np.int64) * 40
    ci = np.arange(m * 40, dtype=np.int32) % n
    v = rng.standard_normal(ci.size)
    U, V = rng.standard_normal((m, r)), rng.standard_normal((r, n))
    for at in (0, 137, ci.size - 1):
        wrong = ci.copy()
        wrong[at] = bad
        with pytest.raises(rt.RtprojError) as e:
            rt.SparseProjector(to_dev(torch, rp), to_dev(torch, wrong), to_dev(torch, v), n, U=to_dev(torch, U), V=to_dev(torch, V),
                               l_max=20, k_max=1)
        assert e.value.code == 1
    rt.SparseProjector(to_dev(torch, rp), to_dev(torch, ci), to_dev(torch, v), n, U=to_dev(torch, U), V=to_dev(torch, V),
                       l_max=20, k_max=1).close()
