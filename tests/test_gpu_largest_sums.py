"""The digit-product kernels (k ≤ 64, and few rows or columns of C) where their
FP32 sums are largest.

A sum of one weight has up to 7 digit pairs at -128 · -128 in each k-entry: an
integer below 2^62 with 53 significant bits holds at most seven such digits, so
7·2^14 an entry, of the 8·2^14 the kernels' bounds allow for.  That is 7/8 of
2^24 over the 128 entries of a slab and of 2^23 over 64.  Digits drawn from -128
and -127 stay within 2% of it and fill the sums' low bits.  The operands are
built from the scales that the call chooses: one larger entry in each row of A
and column of B moves the scale until the others become the integers wanted,
digit for digit.  C must have the oracle's bits, and the residue path's.
"""
import numpy as np
import pytest

from helpers import ensure_built, to_dev
from oracle import ozaki2 as orc


def digits(X):
    """Balanced base-256 digits (in [-128, 127], last axis) of integers below 2^62."""
    biased = X.astype(np.int64).view(np.uint64) + np.uint64(0x8080808080808080)
    return biased[..., None].view(np.uint8).astype(np.int64) - 128


def weight_sums(At, Bt, l0, l1):
    """The largest magnitude of a weight's sum over the entries [l0, l1)."""
    da, db = digits(At[:, l0:l1]), digits(Bt[l0:l1])
    sums = np.zeros((15, At.shape[0], Bt.shape[1]), dtype=np.int64)
    for i in range(8):
        for j in range(8):
            sums[i + j] += da[:, :, i] @ db[:, :, j]
    return int(np.abs(sums).max())


def operands(m, n, k, r):
    """A, B whose scaled integers have the digits -128 and -127 (-120 for the
    last of seven, 53 bits), as many as the scale has room for, but for one entry
    of each row and column; rows and columns of other signs and sizes among them."""
    rng = np.random.default_rng(m + 1000 * n + r)
    shift_a = shift_b = 56
    for nd in (7, 6):
        def entries(rows, cols):
            v = 0.0
            for i in range(nd):
                v = v - rng.choice([128, 120 if i == 0 and nd == 7 else 127], size=(rows, cols)) * 256.0 ** i
            return v
        A0, B0 = entries(m, k), entries(k, n)
        for _ in range(8):
            A, B = A0.copy(), B0.copy()
            A[:, 0] = -2.0 ** shift_a
            B[0, :] = -2.0 ** shift_b
            A[1::3] *= 2.0 ** 40       # another scale, the same integers
            B[:, 2::5] *= 2.0 ** -70
            B[:, 3] *= -1.0            # other digits
            p = orc.prepare(A, B, r)
            da, eb = int(p.d[0]), int(p.e[0])
            if da == 0 and eb == 0:
                return A, B, p, nd
            shift_a, shift_b = shift_a + da, shift_b + eb
            if min(shift_a, shift_b) < 8 * nd:
                break
        shift_a = shift_b = 8 * nd
    raise AssertionError("no scales found")


CASES = [
    ("short", 130, 20, 64, 16, 7), ("short", 130, 35, 64, 14, 7), ("short", 70, 20, 64, 13, 7),
    ("short", 130, 20, 64, 12, 6),
    ("skinny", 130, 20, 500, 16, 7), ("skinny", 20, 130, 500, 16, 7), ("skinny", 130, 16, 300, 14, 7),
    ("skinny", 130, 20, 500, 13, 6), ("skinny", 20, 130, 300, 12, 6),
]


@pytest.mark.parametrize("path,m,n,k,r,pairs", CASES)
def test_the_operands_reach_the_sums(path, m, n, k, r, pairs):
    A, B, p, nd = operands(m, n, k, r)
    assert nd == pairs
    if path == "short":      # one sum over all of k; entry 0 is the scales'
        assert weight_sums(p.At, p.Bt, 0, k) >= 0.98 * (k - 1) * pairs * 2 ** 14
    else:                    # slabs of 128 entries
        assert weight_sums(p.At, p.Bt, 128, 256) >= 0.98 * 128 * pairs * 2 ** 14


@pytest.mark.gpu
@pytest.mark.parametrize("path,m,n,k,r,pairs", CASES)
def test_the_same_bits(path, m, n, k, r, pairs):
    ensure_built()
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2606_06510_gb300 as oz
    A, B, p, _ = operands(m, n, k, r)
    want = orc.evaluate_rows(p, A, B).C.view(np.int64)
    dA, dB = to_dev(A), to_dev(B)
    residues, _ = oz.oz2_dgemm_ex(dA, dB, num_moduli=r)
    assert np.array_equal(residues.cpu().numpy().view(np.int64), want)
    assert np.array_equal(oz.oz2_dgemm(dA, dB, num_moduli=r).cpu().numpy().view(np.int64), want)
    assert oz.oz2_check_device_status() == 0
