"""The float64 QR around the number of columns from which the register form is taken."""
import pytest

import tests.test_gpu_qr_f64 as f64
import workloads
from tests.gpu_common import rt_module, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,l", [(10, 14), (11, 384), (11, 2305), (12, 12), (12, 383), (12, 384), (12, 385), (13, 768), (12, 2305)])
def test_few_columns(m, l):
    torch, rt = torch_cuda(), rt_module()
    f64._check(torch, rt, workloads.haar_spectrum_matrix(m, max(2 * l, 64), 1e-4, 900 + m + l), l, 7)
