"""Short k with flagged rows: recomputed beside the products when they are few,
by the fallback kernel otherwise; the same bits as oz2_dgemm_ex, whose fallback
kernel takes them all."""
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


# Rows are taken beside the products up to a line of sizes (158 of 640 for 200
# columns and k = 64, 47 of 1000 for 4100 and 63): none, one, a group of four and
# its neighbours, both sides of the line, all; columns at a multiple of 32
# and off it, k at the unrolled step's edges and the ends of its range.
@pytest.mark.parametrize("m,n,k,count,r", [
    (640, 96, 64, 0, 12), (640, 97, 64, 1, 12), (640, 31, 64, 4, 12), (640, 33, 64, 5, 12),
    (640, 200, 64, 150, 12), (640, 200, 64, 170, 12),
    (1000, 4100, 63, 7, 8), (1000, 4100, 63, 60, 12), (513, 70, 1, 100, 12), (300, 50, 7, 11, 16), (300, 50, 8, 37, 4),
    (2000, 129, 9, 222, 13), (2000, 1, 17, 117, 12), (40, 3000, 33, 1, 12),
])
@pytest.mark.parametrize("pad", [0, 3])
def test_same_bits_as_the_fallback_kernel(oz, m, n, k, count, r, pad):
    import torch
    A, B = wl.random_matrix(m, k, 1.0, 41 + m + k), wl.random_matrix(k, n, 1.0, 43 + n)
    rng = np.random.default_rng(count)
    for q, i in enumerate(rng.choice(m, count, replace=False)):
        A[i, q % k] = (np.inf, np.nan, -np.inf, 1e300)[q % 4]
    if n > 40:
        B[k // 2, 5] = np.inf
    dA = to_dev(np.pad(A, ((0, pad), (0, 0))))[:m]
    dB = to_dev(np.pad(B, ((0, pad), (0, 0))))[:k]
    want, _ = oz.oz2_dgemm_ex(dA, dB, num_moduli=r)
    rows = oz.oz2_get_stats()["fallback_rows"]
    got = oz.oz2_dgemm(dA, dB, num_moduli=r)
    assert oz.oz2_get_stats()["fallback_rows"] == rows
    assert torch.equal(got.t().contiguous().view(torch.int64), want.t().contiguous().view(torch.int64))
    assert oz.oz2_check_device_status() == 0
