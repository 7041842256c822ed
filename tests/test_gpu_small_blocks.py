"""The sizes at which the scan and the deconstruction change their blocks.

The scan gives a thread of A 64, 32, 16 or 8 k-entries and a warp of B 1024
or 256, by the blocks the operand makes; its exponents are compared with
numpy's frexp at sizes that take each length, and at remainders of the load
batches.  The deconstruction takes blocks of a quarter of the rows up to one
full tile per SM; the planes on both sides of that line must agree.
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


@pytest.mark.parametrize("m,n,k", [
    (1, 1, 1), (257, 9, 7), (3, 5, 257), (300, 40, 1025), (520, 2, 20000), (2, 700, 2047), (4096, 9, 1280), (9, 9728, 31),
])
def test_scan_exponents(oz, m, n, k):
    A, B = wl.random_matrix(m, k, 3.0, 300 + k), wl.random_matrix(k, n, 3.0, 400 + k)
    A[m // 2, k - 1] *= 2.0 ** 20     # decisive entries at the ends of the runs
    B[k - 1, n // 2] *= 2.0 ** 20
    pad = np.zeros((k + 1, n))
    for b in (to_dev(B), to_dev(np.vstack([pad[:1], B]))[1:]):  # 16-byte aligned columns, and not
        ra, cb, rf, cf = oz.oz2_scan(to_dev(A), b, flags=oz.FLAG_NO_FALLBACK)
        assert np.array_equal(ra.cpu().numpy(), np.frexp(np.abs(A).max(axis=1))[1])
        assert np.array_equal(cb.cpu().numpy(), np.frexp(np.abs(B).max(axis=0))[1])
        assert not rf.any() and not cf.any()


@pytest.mark.parametrize("r", [6, 12, 16])
def test_planes_agree_across_the_block_rule(oz, r):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    m = sms // 8 * 128                 # half the SMs' worth of 32-row tiles in each operand
    A, B = to_dev(wl.random_matrix(m, 100, 1.0, 501)), to_dev(wl.random_matrix(100, m + 256, 1.0, 502))
    e = torch.full((m + 256,), 45, dtype=torch.int32, device="cuda")
    f = torch.zeros(m + 256, dtype=torch.uint8, device="cuda")
    pa, pb = oz.oz2_deconstruct(A, B[:, :m], e[:m], e[:m], f[:m], f[:m], r)
    pa2, pb2 = oz.oz2_deconstruct(A, B, e[:m], e, f[:m], f, r)
    assert torch.equal(pa, pa2) and torch.equal(pb, pb2[:m // 128])
