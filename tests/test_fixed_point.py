"""CPU pins of the fixed-point arithmetic of the float64 block products (csrc/fixed.cuh),
restated here in integers: the encoding rounds to 2^-57 of its scale whatever the shift, its
two parts fit their bounds, and a 64-term dot product from three integer products per term is
within 64 (2^-57 + 2^-57 + 2^-56) of the largest product of the exact one."""
import random
import struct
from fractions import Fraction

import pytest


def exponent(v):
    return (struct.unpack("<Q", struct.pack("<d", v))[0] >> 52) & 0x7FF


def encode(v, E):
    b = struct.unpack("<Q", struct.pack("<d", v))[0]
    hi, lo = b >> 32, b & 0xFFFFFFFF
    sh = (((E + 4) << 20) - (hi & 0x7FF00000)) >> 20
    t, low = ((hi << 11 | lo >> 21) & 0xFFFFFFFF) | 0x80000000, (lo << 11) & 0xFFFFFFFF
    h = t >> sh if sh < 32 else 0
    part = ((t << 32 | low) >> min(sh, 32)) & 0xFFFFFFFF
    r = max(sh, 32) - 29
    part = ((part >> r if r < 32 else 0) + 1) >> 1
    s = -1 if hi >> 31 else 1
    return h * s, part * s


@pytest.mark.parametrize("shift", [0, 1, 3, 4, 27, 28, 29, 31, 32, 33, 55, 56, 57, 59, 60, 63, 64, 200])
def test_encoding_rounds_to_nearest_at_every_shift(shift):
    rng = random.Random(shift)
    lean = 0.0
    for k in range(2000):
        v = rng.choice([-1, 1]) * (1 + rng.getrandbits(52) * 2.0 ** -52) * 2.0 ** rng.randint(-300, 300)
        if k == 0:
            v = float.fromhex("0x1.fffffffffffffp+3")
        E = exponent(v) + shift
        h, l = encode(v, E)
        err = h * 2 ** 28 + l - Fraction(v) * Fraction(2) ** (1078 - E)
        assert abs(err) <= Fraction(1, 2)
        assert abs(h) < 2 ** 28 and abs(l) <= 2 ** 28
        lean += float(err) * (1 if v > 0 else -1)
    # the errors have no lean: their sum over 2000 draws is within 8 of its standard
    # deviations (1 / sqrt(12) each) of what halves rounded up give (half a unit with
    # probability 2^-k where k bits are dropped); shifts that drop every bit have no spread
    if shift <= 55:
        k = max(0, shift - 3)
        assert abs(lean - (1000 * 2.0 ** -k if k else 0.0)) <= 8 * (2000 / 12) ** 0.5
    assert encode(0.0, 128) == (0, 0) and encode(-0.0, 1023) == (0, 0)


@pytest.mark.parametrize("spread", [0, 10, 60])
def test_dot_product_of_64_terms(spread):
    rng = random.Random(spread)
    for _ in range(50):
        a = [rng.gauss(0, 1) * 2.0 ** -rng.randint(0, spread) for _ in range(64)]
        b = [rng.gauss(0, 1) * 2.0 ** -rng.randint(0, spread) for _ in range(64)]
        Ea, Eb = max(map(exponent, a)), max(map(exponent, b))
        hh, mid = 0, 2 ** 27
        for x, y in zip(a, b):
            (h, l), (g, m) = encode(x, Ea), encode(y, Eb)
            hh += h * g
            mid += h * m + l * g
            assert abs(hh) < 2 ** 63 and abs(mid) < 2 ** 63
        got = Fraction(hh + (mid >> 28)) * Fraction(2) ** (Ea + Eb - 2100)
        exact = sum(Fraction(x) * Fraction(y) for x, y in zip(a, b))
        scale = Fraction(2) ** (Ea - 1022) * Fraction(2) ** (Eb - 1022)
        assert abs(got - exact) <= 64 * scale * (Fraction(2, 2 ** 57) + Fraction(1, 2 ** 56))
