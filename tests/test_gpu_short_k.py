"""C from base-256 digit products (k ≤ 64, oz2_dgemm and oz2_dgemm_host).

The path forms the same integer X as the residues do, so C must equal the
residue path's (oz2_dgemm_ex) bit for bit: at the edges of its tiles (128
rows, 16 columns) and K-steps (16 entries), over the moduli counts (with the
128- and 160-bit roundings), strides and special rows, and with the sums at
their largest (every digit -128).
"""
import numpy as np
import pytest

import workloads as wl
from helpers import ensure_built, to_dev
from oracle import ozaki2 as orc

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


def bits(t):
    """float64 bits, with one pattern for every NaN (its payload is not part of the result)."""
    x = t.cpu().numpy()
    return np.where(np.isnan(x), np.nan, x).view(np.int64)


def check(oz, A, B, r):
    want, _ = oz.oz2_dgemm_ex(A, B, num_moduli=r)
    got = oz.oz2_dgemm(A, B, num_moduli=r)
    assert np.array_equal(bits(got), bits(want))
    assert oz.oz2_check_device_status() == 0
    return got


@pytest.mark.parametrize("m,n,k,r", [
    (1, 1, 1, 12), (128, 16, 16, 12), (129, 17, 17, 13), (127, 15, 64, 16), (300, 333, 63, 12), (1000, 2100, 48, 12),
    (64, 4000, 33, 14), (4000, 40, 64, 4), (513, 257, 64, 1), (260, 250, 31, 6), (140, 30, 64, 3), (2, 70, 65, 12),
])
def test_matches_the_residue_path(oz, m, n, k, r):
    for phi in (0.5, 4.0):
        A, B = wl.random_matrix(m, k, phi, 40 + m), wl.random_matrix(k, n, phi, 50 + n)
        check(oz, to_dev(A), to_dev(B), r)


def test_oracle_special_rows_and_strides(oz):
    import torch
    m, n, k = 200, 150, 60
    A, B = np.array(wl.random_matrix(m, k, 2.0, 61)), np.array(wl.random_matrix(k, n, 2.0, 62))
    A[3] = 0.0
    A[5] *= 2.0 ** 300
    A[7, 2] = np.inf
    A[9] *= 2.0 ** -100
    A[11, 1:] = 0.0
    B[:, 4] = 0.0
    B[:, 6] *= 2.0 ** -300
    B[5, 8] = np.nan
    B[:, 17] = 5e-324
    for r in (12, 15):
        want = orc.oz2_dgemm(A, B, r).C
        big = torch.zeros((k, m + 3), dtype=torch.float64, device="cuda").t()   # odd leading dimensions
        big[:m] = to_dev(A)
        bigb = torch.zeros((n, k + 1), dtype=torch.float64, device="cuda").t()
        bigb[:k] = to_dev(B)
        out = torch.full((n, m + 5), -7.0, dtype=torch.float64, device="cuda").t()
        oz.oz2_dgemm(big[:m], bigb[:k], out[:m], num_moduli=r)
        got = out[:m].cpu().numpy()
        assert np.array_equal(bits(out[:m]), np.where(np.isnan(want), np.nan, want).view(np.int64))
        num = ~np.isnan(got)
        assert np.array_equal(np.signbit(got[num]), np.signbit(want[num]))
        assert (out[m:].cpu().numpy() == -7.0).all()                            # C's pad rows stay
        assert np.array_equal(np.nan_to_num(oz.oz2_dgemm_host(A, B, num_moduli=r)), np.nan_to_num(want))


def test_subnormal_operands(oz):
    A = np.array(wl.random_matrix(150, 40, 1.0, 63)) * 2.0 ** -1060
    B = np.array(wl.random_matrix(40, 70, 1.0, 64)) * 2.0 ** 1000
    check(oz, to_dev(A), to_dev(B), 12)


def test_sums_at_their_largest(oz):
    """Entries whose scaled integers have every low digit -128 (64 products of
    2^14 from up to 8 digit pairs: 2^23 in one FP32 sum)."""
    v = -sum(128 * 256 ** i for i in range(6))
    A = np.full((130, 64), float(v))
    B = np.full((64, 20), float(v))
    A[1::2] *= 3.0
    B[:, 3] *= -1.0
    for r in (12, 13, 16):
        check(oz, to_dev(A), to_dev(B), r)
