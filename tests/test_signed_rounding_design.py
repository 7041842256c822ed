"""The two's complement rounding of X·2^E (reconstruction, short-k and skinny
kernels) against the oracle's correctly rounded unscale, on the CPU.

The kernels round the signed word under X's redundant sign bits, a sticky bit
for the rest in bit 0, with the hardware's signed conversion (Python's correctly
rounded int → float here) and never take |X|; 160-bit values whose top word is
more than a sign drop their lowest word into the sticky bit first.
"""
import random
import struct

import pytest

from oracle import ozaki2 as orc

M32, M64 = (1 << 32) - 1, (1 << 64) - 1


def bits_of(x: float) -> int:
    return struct.unpack("<Q", struct.pack("<d", x))[0]


def signed(v: int, n: int) -> int:
    v &= (1 << n) - 1
    return v - (1 << n) if v >> (n - 1) else v


def scaled(top: int, e: int) -> int:
    """The bits of float(top) with e added to the exponent field."""
    return (bits_of(float(top)) + (e << 52)) & M64


def finish_signed(w3, w2, w1, w0, E):
    sg = M32 if w3 >> 31 else 0
    y3, y2 = w3 ^ sg, w2 ^ sg
    if (y3 | y2) == 0 and (w1 ^ sg) >> 31 == 0:
        x = signed((w1 << 32) | w0, 64)
        if x == 0:
            return 0
        return None if E < -1022 or E > 1023 - 64 else scaled(x, E)
    sh = (32 - y3.bit_length() if y3 else 64 - y2.bit_length()) - 1
    ex = E + 64 - sh
    if ex < -1022 - 62 or ex > 1021 - 62:
        return None  # the general routine
    x3, x2, x1, x0 = (w2, w1, w0, 0) if sh >= 32 else (w3, w2, w1, w0)
    sp = sh & 31
    th = ((((x3 << 32) | x2) << sp) >> 32) & M32
    tl = ((((x2 << 32) | x1) << sp) >> 32) & M32
    sticky = 1 if (((x1 << sp) & M32) | x0) else 0
    top = signed((th << 32) | tl | sticky, 64)
    assert 1 << 62 <= abs(top) <= 1 << 63
    return scaled(top, ex)


def finish_signed160(w, E):
    big = signed(w[4], 32) != (-1 if w[3] >> 31 else 0)
    if big:
        return finish_signed(w[4], w[3], w[2], w[1] | (1 if w[0] else 0), E + 32)
    return finish_signed(w[3], w[2], w[1], w[0], E)


def check(X, E):
    words = [(X >> (32 * i)) & M32 for i in range(5)]
    want = bits_of(orc.unscale_one(X, E)) if X else 0
    results = [finish_signed160(words, E)]
    if -(1 << 127) <= X < 1 << 127:
        results.append(finish_signed(words[3], words[2], words[1], words[0], E))
    for got in results:
        assert got is None or got == want, (X, E, got, want)
    return results[0] is not None


@pytest.mark.parametrize("bits", [159, 127])
def test_random_values_every_range(bits):
    rnd = random.Random(bits)
    fast = 0
    for _ in range(40_000):
        L = rnd.randint(1, bits)
        X = rnd.getrandbits(L) | (1 << (L - 1))
        fast += check(-X if rnd.random() < 0.5 else X, rnd.randint(-1250, 1030 - L))
    assert fast > 25_000


def test_ties_powers_and_word_edges():
    rnd = random.Random(7)
    for _ in range(8_000):
        L = rnd.randint(55, 158)
        base, half = (rnd.getrandbits(53) | (1 << 52)) << (L - 53), 1 << (L - 54)
        for X in (base + half, base + half - 1, base + half + 1, base + 1, base):
            for s in (1, -1):
                assert check(s * X, rnd.randint(-1000, 850 - L))
    for L in range(0, 158):
        for X in (1 << L, (1 << L) - 1, (1 << L) + 1, (1 << L) + (1 << (L // 2)), (1 << L) - (1 << (L // 3))):
            for E in (-1200, -1022, -300, 0, 700):
                check(X, E)
                check(-X, E)
    check(0, 0)
