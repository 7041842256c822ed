"""C of few rows or columns from base-256 digits formed on chip (oz2_dgemm and
oz2_dgemm_host).

The path forms the same integer X as the residues do, so C must equal the
residue path's (oz2_dgemm_ex) bit for bit: at the edges of its tiles (128 rows,
16 columns), chunks (32 entries) and slabs (128), with either operand tall,
over the moduli counts, strides and special rows, with runs of work that end
inside a row block, and with the sums at their largest (2^24).
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


@pytest.mark.parametrize("m,n,k,r", [
    (1, 1, 65, 12), (128, 16, 128, 12), (129, 17, 129, 13), (127, 15, 255, 16), (1, 300, 1000, 12), (300, 1, 97, 8),
    (5000, 33, 4100, 12), (64, 3000, 777, 14), (1000, 32, 333, 4), (3, 5, 70000, 12), (20, 130, 20000, 6),
    (16, 16, 65, 1), (2100, 48, 160, 15), (65, 64, 300, 12), (70, 80, 300, 16), (100, 81, 200, 16), (33, 90, 200, 6),
])
def test_matches_the_residue_path(oz, m, n, k, r):
    for phi in (0.5, 3.0):
        A, B = wl.random_matrix(m, k, phi, 70 + m), wl.random_matrix(k, n, phi, 80 + n)
        check(oz, to_dev(A), to_dev(B), r)


@pytest.mark.parametrize("shape", [(200, 30, 300), (30, 200, 300)])
def test_oracle_special_rows_and_strides(oz, shape):
    import torch
    m, n, k = shape
    A, B = np.array(wl.random_matrix(m, k, 2.0, 91)), np.array(wl.random_matrix(k, n, 2.0, 92))
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


def test_host_column_blocks(oz):
    m, n, k = 40, 3000, 2000
    A, B = np.array(wl.random_matrix(m, k, 1.0, 93), order="F"), np.array(wl.random_matrix(k, n, 1.0, 94), order="F")
    want, _ = oz.oz2_dgemm_ex(to_dev(A), to_dev(B))
    assert np.array_equal(oz.oz2_dgemm_host(A, B), want.cpu().numpy())


@pytest.mark.parametrize("m,n,k", [(4100, 33, 4095), (130, 80, 130000), (16800, 3, 1001)])
def test_plus_one_pass_on_chip(oz, m, n, k):
    """A larger than L2 (2^24 entries): its magnitude codes are formed on chip as
    well.  Rows that are zero, flagged or far down in scale, an odd ld."""
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(97)
    A = torch.randn((k, m + 1), dtype=torch.float64, device="cuda", generator=g).t()[:m]
    B = torch.randn((n, k), dtype=torch.float64, device="cuda", generator=g).t()
    A[5] = 0.0
    A[7] *= 2.0 ** 300
    A[9, 3] = float("inf")
    A[11] *= 2.0 ** -90
    B[:, 1] = 0.0
    check(oz, A, B, 12)


def test_subnormal_operands(oz):
    A = np.array(wl.random_matrix(150, 400, 1.0, 95)) * 2.0 ** -1060
    B = np.array(wl.random_matrix(400, 20, 1.0, 96)) * 2.0 ** 1000
    check(oz, to_dev(A), to_dev(B), 12)


def test_sums_at_their_largest(oz):
    """Entries whose scaled integers have every low digit -128: 8 digit pairs ·
    128 entries · 2^14 = 2^24 in one FP32 sum, over several slabs."""
    v = -sum(128 * 256 ** i for i in range(6))
    A = np.full((130, 500), float(v))
    B = np.full((500, 20), float(v))
    A[1::2] *= 3.0
    B[:, 3] *= -1.0
    for r in (12, 13, 16):
        check(oz, to_dev(A), to_dev(B), r)
