"""oz2_dgemm_host splits the residue GEMM as oz2_plan's host_kparts says, also
where oz2_dgemm takes parts of its own.

A split shows in the launches: its parts' residues are folded by one more
kernel.  Beside that a host call of one column block, whose A arrives in one
piece, launches three kernels more than oz2_dgemm (B's scan, flags and magnitude
planes run apart from A's).
"""
import numpy as np
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


@pytest.mark.parametrize("m,n,k,r,planned,own", [
    (515, 81, 3815, 13, 2, 1), (1282, 86, 4663, 13, 1, 2), (197, 130, 6151, 6, 2, 2), (700, 200, 700, 12, 1, 1),
])
def test_host_call_takes_the_planned_parts(oz, m, n, k, r, planned, own):
    plan = oz.oz2_plan(m, n, k, r)
    assert plan["host_widths"] == [n]
    assert min(plan["host_kparts"][0], 2) == planned
    A = np.array(wl.random_matrix(m, k, 1.0, 700 + m), order="F")
    B = np.array(wl.random_matrix(k, n, 1.0, 800 + n), order="F")
    dA, dB = to_dev(A), to_dev(B)

    def launches(call):
        call()
        oz.oz2_get_stats()
        got = call()
        return got, oz.oz2_get_stats()["kernel_launches"]

    want, device = launches(lambda: oz.oz2_dgemm(dA, dB, num_moduli=r))
    got, host = launches(lambda: oz.oz2_dgemm_host(A, B, num_moduli=r))
    assert host - device == 3 + planned - own
    assert np.array_equal(got.view(np.int64), want.cpu().numpy().view(np.int64))
    assert oz.oz2_check_device_status() == 0
