"""CPU pins of the split of the fixed-point tiles (csrc/fixed.cuh, fx_encode_even): the same value
as before with a low part of either sign, so that the part of a product that is left out has no
lean, and sums of 64 and 128 terms that stay in 64 bits."""
import random
import struct
from fractions import Fraction

import pytest

B = 28


def bits(v):
    return struct.unpack("<Q", struct.pack("<d", v))[0]


def exponent(v):
    return (bits(v) >> 52) & 0x7FF


def encode_even(v, E):
    hi, lo = bits(v) >> 32, bits(v) & 0xFFFFFFFF
    sh = ((((E + 32 - B) << 20) - (hi & 0x7FF00000)) & 0xFFFFFFFF) >> 20
    t, low = ((hi << 11 | lo >> 21) & 0xFFFFFFFF) | 0x80000000, (lo << 11) & 0xFFFFFFFF
    h = t >> sh if sh < 32 else 0
    part = ((t << 32 | low) >> min(sh, 32)) & 0xFFFFFFFF
    r = max(sh, 32) - B - 1
    part = ((part >> r if r < 32 else 0) + 1) >> 1
    s = -1 if hi >> 31 else 1
    h, l = h * s, part * s
    c = (l + (1 << (B - 1))) >> B
    return h + c, l - (c << B)


@pytest.mark.parametrize("shift", [0, 1, 3, 4, 27, 28, 29, 31, 32, 33, 55, 57, 60, 64, 200])
def test_values_and_bounds(shift):
    rng = random.Random(shift)
    for k in range(1000):
        v = rng.choice([-1, 1]) * (1 + rng.getrandbits(52) * 2.0 ** -52) * 2.0 ** rng.randint(-300, 300)
        if k == 0:
            v = float.fromhex("0x1.fffffffffffffp+3")
        E = exponent(v) + shift
        h, l = encode_even(v, E)
        assert abs(h * 2 ** B + l - Fraction(v) * Fraction(2) ** (1022 + 2 * B - E)) <= Fraction(1, 2)
        assert abs(h) <= 2 ** B and abs(l) <= 2 ** (B - 1)
    assert encode_even(0.0, 128) == (0, 0)


def test_sums_of_the_largest_values_fit():
    h, l = 2 ** B, 2 ** (B - 1)
    assert 64 * h * h + (64 * 2 * h * l >> B) < 2 ** 63 and 64 * 2 * h * l + 2 ** (B - 1) < 2 ** 63
    # 128 terms under a bit of headroom in both operands
    assert 128 * (h // 2) ** 2 < 2 ** 63 and 128 * 2 * (h // 2) * l < 2 ** 63


def test_what_is_left_out_has_no_lean():
    rng = random.Random(1)
    n, left = 20000, 0
    for _ in range(n):
        (_, l), (_, m) = encode_even(rng.uniform(0.1, 1.0), 1023), encode_even(rng.uniform(0.1, 1.0), 1023)
        left += l * m
    # uniform parts of size 2^(B - 1): products of variance 2^(4 B - 4) / 9; with parts cut towards
    # zero their mean would be 2^(2 B - 2), n^0.5 / 4 * 3 = 106 of these deviations
    assert abs(left) <= 6 * n ** 0.5 * 2 ** (2 * B - 2) / 3
