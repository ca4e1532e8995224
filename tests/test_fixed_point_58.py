"""CPU pins of the 58-bit fixed point of the float64 block products (csrc/fixed.cuh, parts of
29 bits): values are rounded at 2^-59 of the scale and exact within 2^-5 of it, and the sums of
a lane (16 terms for a row, 8 for a column) and of eight lanes stay in 64 bits."""
import random
import struct
from fractions import Fraction

import pytest

B = 29


def bits(v):
    return struct.unpack("<Q", struct.pack("<d", v))[0]


def exponent(v):
    return (bits(v) >> 52) & 0x7FF


def encode(v, E):
    hi, lo = bits(v) >> 32, bits(v) & 0xFFFFFFFF
    sh = ((((E + 32 - B) << 20) - (hi & 0x7FF00000)) & 0xFFFFFFFF) >> 20
    t, low = ((hi << 11 | lo >> 21) & 0xFFFFFFFF) | 0x80000000, (lo << 11) & 0xFFFFFFFF
    h = t >> sh if sh < 32 else 0
    part = ((t << 32 | low) >> min(sh, 32)) & 0xFFFFFFFF
    r = max(sh, 32) - B - 1
    part = ((part >> r if r < 32 else 0) + 1) >> 1
    s = -1 if hi >> 31 else 1
    return h * s, part * s


@pytest.mark.parametrize("shift", [0, 1, 2, 4, 5, 6, 28, 29, 30, 31, 32, 57, 58, 59, 63, 64, 1500])
def test_encoding(shift):
    rng = random.Random(shift)
    for k in range(1000):
        v = rng.choice([-1, 1]) * (1 + rng.getrandbits(52) * 2.0 ** -52) * 2.0 ** rng.randint(-300, 300)
        if k == 0:
            v = float.fromhex("0x1.fffffffffffffp+3")
        E = exponent(v) + shift
        h, l = encode(v, E)
        err = abs(h * 2 ** B + l - Fraction(v) * Fraction(2) ** (1022 + 2 * B - E))
        assert err <= (0 if shift <= 5 else Fraction(1, 2))
        assert abs(h) < 2 ** B and abs(l) <= 2 ** B
    assert encode(0.0, 1023) == (0, 0) and encode(-0.0, 1500) == (0, 0)


def test_sums_of_the_largest_values_fit():
    h, l = 2 ** B - 1, 2 ** B
    hh, mid = 16 * h * h, 16 * 2 * h * l + 2 ** (B - 1)                 # a row: 16 passes
    assert hh + (mid >> B) < 2 ** 63 and mid < 2 ** 63
    g, m = 2 ** (B - 1) - 1, 2 ** B                                     # the row's x: an exponent more
    hh, mid = 8 * h * g, 8 * (h * m + l * g) + 2 ** (B - 1)             # a column: 8 rows,
    assert mid < 2 ** 63 and 8 * (hh + (mid >> B)) < 2 ** 63            # then 8 lanes


@pytest.mark.parametrize("spread", [0, 5, 60])
def test_column_of_64_terms(spread):
    rng = random.Random(spread)
    for _ in range(50):
        a = [rng.gauss(0, 1) * 2.0 ** -rng.randint(0, spread) for _ in range(64)]
        b = [rng.gauss(0, 1) * 2.0 ** -rng.randint(0, spread) for _ in range(64)]
        Ea, Eb = max(map(exponent, a)), max(map(exponent, b)) + 1
        total = 0
        for lane in range(8):
            hh, mid = 0, 2 ** (B - 1)
            for x, y in zip(a[8 * lane:8 * lane + 8], b[8 * lane:8 * lane + 8]):
                (h, l), (g, m) = encode(x, Ea), encode(y, Eb)
                hh += h * g
                mid += h * m + l * g
            total += hh + (mid >> B)
        got = Fraction(total) * Fraction(2) ** (Ea + Eb - 2102)
        exact = sum(Fraction(x) * Fraction(y) for x, y in zip(a, b))
        scale = Fraction(2) ** (Ea + Eb - 2044)
        # relative to the scales, b's doubled by its exponent: per term two encodings at 2^-59 and the
        # part left out at 2^-58; per lane half a unit of 2^-58
        assert abs(got - exact) <= scale * (64 * Fraction(2, 2 ** 58) + 8 * Fraction(1, 2 ** 59))
