"""The residue GEMM's ordering of a unit's products, bit for bit.

For k > 128 the kernel fills the two accumulators of a modulus apart: a
nonsquare modulus one after the other, a square one in three phases whose
first and last cover the first five k-blocks; the residue then travels from
K-slab to K-slab in registers.  The sizes sit at the edges of those phases
(four to seven k-blocks), of the K-slabs (4096 and 32768 k-entries) and of
the tiles (of 64 columns where those fill one wave), and the result is compared with the CUDA-core twin, which sums the
same plane products in sequential k order.
"""
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
    (1, 1, 129, 16), (130, 260, 256, 8), (257, 17, 512, 16), (300, 255, 640, 8), (256, 256, 641, 8),
    (129, 258, 768, 16), (64, 33, 896, 12), (257, 300, 4096, 8), (40, 272, 4097, 16), (130, 20, 8200, 8),
    (16, 24, 32768, 8), (33, 16, 33409, 8),
    # 64-column tiles, up to one wave of the CTA pairs, and just past it
    (256, 384, 200, 12), (256, 385, 200, 12), (130, 65, 300, 16), (100, 127, 4200, 3), (20, 1279, 256, 3),
])
def test_phases_match_the_sequential_twin(oz, m, n, k, r):
    import torch
    A, B = to_dev(wl.random_matrix(m, k, 1.0, 8100 + k)), to_dev(wl.random_matrix(k, n, 1.0, 8200 + k))
    d = torch.full((m,), 50, dtype=torch.int32, device="cuda")
    e = torch.full((n,), 50, dtype=torch.int32, device="cuda")
    rf, cf = (torch.zeros(x, dtype=torch.uint8, device="cuda") for x in (m, n))
    pa, pb = oz.oz2_deconstruct(A, B, d, e, rf, cf, r)
    got = oz.oz2_residue_gemm(pa, pb, m, n, k, r)
    want = oz.oz2_residue_gemm(pa, pb, m, n, k, r, simt=True)
    assert torch.equal(got, want)
    assert oz.oz2_check_device_status() == 0
