"""oz2_dgemm takes its own parts of k (residue GEMM and magnitude GEMM), where
oz2_dgemm_ex keeps to oz2_plan's: the same bits at sizes where the two differ,
and at ragged last parts."""
import pytest

import workloads as wl
from helpers import ensure_built, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def oz():
    ensure_built()
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2606_06510_gb300 as oz
    oz.lib()
    return oz


@pytest.mark.parametrize("m,n,k,r", [
    (1000, 777, 1333, 12),      # the magnitude GEMM unsplit instead of in two parts
    (256, 250, 30000, 12),      # six parts instead of twelve
    (1024, 1000, 20001, 12),    # parts where the plan has none
    (300, 400, 20000, 14), (513, 255, 9000, 6), (100, 100, 70000, 16),
])
def test_same_bits_as_the_planned_call(oz, m, n, k, r):
    import torch
    A, B = to_dev(wl.random_matrix(m, k, 1.0, 600 + m)), to_dev(wl.random_matrix(k, n, 1.0, 700 + n))
    want, _ = oz.oz2_dgemm_ex(A, B, num_moduli=r)
    got = oz.oz2_dgemm(A, B, num_moduli=r)
    assert torch.equal(got.t().contiguous().view(torch.int64),
                       want.t().contiguous().view(torch.int64))
    assert oz.oz2_check_device_status() == 0
