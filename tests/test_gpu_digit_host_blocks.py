"""oz2_dgemm_host in several column blocks on the digit-product paths (few rows
of C, and k ≤ 64): each block starts inside B, its exponents, flags and C, shares
the scratch with the block before, and decides anew which operand is the tall
one; flagged rows and columns go to the fallback block by block.  The bits are
those of oz2_dgemm_ex on device copies, which forms residues in one piece."""
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


def bits(x):
    """float64 bits, with one pattern for every NaN."""
    return np.where(np.isnan(x), np.nan, x).view(np.int64)


@pytest.mark.parametrize("m,n,k,r,widths", [
    (40, 8000, 500, 12, [6400, 1600]),
    (80, 12000, 128, 16, [4864, 3584, 3552]),
    (40, 4888, 366, 8, [4864, 24]),             # the last block is taller than wide
    (66, 3602, 399, 16, [3584, 18]),
    (700, 3001, 64, 12, None), (1500, 1030, 33, 6, None),   # k ≤ 64
])
@pytest.mark.parametrize("special", [False, True])
def test_blocks(oz, m, n, k, r, widths, special):
    plan = oz.oz2_plan(m, n, k, r)["host_widths"]
    assert len(plan) > 1 and (widths is None or plan == widths)
    A = np.array(wl.random_matrix(m, k, 1.0, 900 + m), order="F")
    B = np.array(wl.random_matrix(k, n, 1.0, 950 + n), order="F")
    if special:
        A[m // 2] *= 2.0 ** 300
        A[3] = 0.0
        A[m - 1, 2] = np.inf
        for c in np.cumsum([0] + plan[:-1]):      # in each block
            B[:, c] *= 2.0 ** -300
            B[:, c + 5] = 0.0
            B[1, c + 9] = np.nan
        B[:, n - 1] *= 2.0 ** 290
    want, _ = oz.oz2_dgemm_ex(to_dev(A), to_dev(B), num_moduli=r)
    out = np.full((m, n), -7.0, order="F")
    assert np.array_equal(bits(oz.oz2_dgemm_host(A, B, out, num_moduli=r)), bits(want.cpu().numpy()))
    assert oz.oz2_check_device_status() == 0
