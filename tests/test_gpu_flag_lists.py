"""oz2_dgemm's fallback lists come from the flags kernel, where oz2_dgemm_ex
lists the flagged rows and columns in a launch of its own: the same bits."""
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


# A block of 1024 threads makes each operand's list, eight entries a thread at
# a time: below, at and past one pass of the block and of the batch.
@pytest.mark.parametrize("m,n,k,rows,cols", [
    (1, 1, 3, [0], []), (3, 2, 40, [0, 2], [1]),
    (1023, 1025, 130, [0, 511, 1022], [0, 1024]),
    (8192, 40, 48, [0, 1024, 8191], []), (8200, 33, 200, list(range(7000, 8200)), [0, 32]),
    (33, 8193, 200, [], [0, 8191, 8192]), (300, 200, 5000, [], []),
])
def test_same_bits_as_the_listing_launch(oz, m, n, k, rows, cols):
    import torch
    A, B = wl.random_matrix(m, k, 1.0, 31 + m), wl.random_matrix(k, n, 1.0, 37 + n)
    for q, i in enumerate(rows):
        if q % 2:
            A[i, q % k] = np.inf if q % 4 == 1 else np.nan
        else:
            A[i, :] *= 2.0 ** (400 if len(rows) < m / 2 else 0)
    for j in cols:
        B[(j + 1) % k, j] = -np.inf
    dA, dB = to_dev(A), to_dev(B)
    want, _ = oz.oz2_dgemm_ex(dA, dB, num_moduli=12)
    want_stats = oz.oz2_get_stats()
    got = oz.oz2_dgemm(dA, dB, num_moduli=12)
    stats = oz.oz2_get_stats()
    assert torch.equal(got.t().contiguous().view(torch.int64), want.t().contiguous().view(torch.int64))
    assert (stats["fallback_rows"], stats["fallback_cols"]) == (want_stats["fallback_rows"], want_stats["fallback_cols"])
    assert oz.oz2_check_device_status() == 0
