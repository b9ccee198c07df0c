"""Integer forms of the digit scheme's conversions (gemm_f64.cu), restated with Python integers against exact rationals.

to_fixed: x 2^(56 - e) rounded to an integer (ties to even) from the FP64 significand; its eight digits; fixed_scaled:
(hi 2^-31 + lo 2^-63) 2^s rounded once to FP64; and the group sums over K = 384.  No GPU is needed."""
import random
import struct
from fractions import Fraction

import pytest


def _bits(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0]


def _exponent(m):
    ex = m >> 52
    return ex - 1022 if ex > 0 else m.bit_length() - 1074


def _to_fixed(x, e):
    b = _bits(x)
    ex, m = (b >> 52) & 0x7FF, b & ((1 << 52) - 1)
    m, ex = (m | 1 << 52, ex) if ex else (m, 1)
    sh = ex - 1019 - e
    if sh >= 0:
        assert sh <= 3
        X = m << sh
    else:
        r = min(-sh, 54)
        X = (m + ((1 << (r - 1)) - 1) + ((m >> r) & 1)) >> r
    return -X if b >> 63 else X


def _round_even(f):
    n = f.numerator // f.denominator
    r = f - n
    return n + (1 if r > Fraction(1, 2) or (r == Fraction(1, 2) and n % 2) else 0)


@pytest.mark.parametrize("kind", range(4))
def test_fixed_point_words_and_digits(kind):
    rng = random.Random(kind)
    for _ in range(5000):
        x = (rng.uniform(-1, 1) * 2.0 ** rng.randint(-80, 3), rng.uniform(-1, 1) * 2.0 ** rng.randint(-1000, 1000),
             rng.randint(1, 2**20) * 2.0 ** rng.randint(-1074, -1040),
             (rng.randrange(1, 1 << 10) + 0.5) * 2.0**-57 * rng.choice((-1, 1)))[kind]
        if x == 0:
            continue
        e0 = _exponent(_bits(abs(x)))
        assert Fraction(2) ** (e0 - 1) <= abs(Fraction(x)) < Fraction(2) ** e0
        e = max(e0 + rng.choice((0, 0, 1, 20, 54, 55, 56, 57, 58, 100)), -960)
        X = _to_fixed(x, e)
        assert abs(X) == _round_even(abs(Fraction(x)) * Fraction(2) ** (56 - e)) <= 2**56
        # the digits as the fields of X with 64 added at every digit but the first
        Y = X + sum(64 << (7 * q) for q in range(7))
        digits = [Y >> 49] + [((Y >> (7 * (7 - p))) & 127) - 64 for p in range(1, 8)]
        assert abs(digits[0]) <= 128 and all(abs(d) <= 64 for d in digits[1:])
        assert sum(d << (7 * (7 - p)) for p, d in enumerate(digits)) == X


def _fixed_scaled(hi, lo, s):
    neg = hi < 0
    alo = (-lo) & 0xFFFFFFFF if neg else lo
    ahi = (~hi + (lo == 0)) if neg else hi
    sticky = False
    if ahi:
        lz = 64 - ahi.bit_length()
        t = (ahi << lz) & ((1 << 64) - 1)
        if lz >= 32:
            t |= alo << (lz - 32)
        else:
            t |= alo >> (32 - lz)
            sticky = (alo << lz) & 0xFFFFFFFF != 0
    elif alo:
        lz = 64 + 32 - alo.bit_length()
        t = alo << (lz - 32)
    else:
        return 0.0
    m, rem = t >> 11, t & 0x7FF
    m += rem > 0x400 or (rem == 0x400 and (sticky or m & 1))
    m += (1055 - lz + s - 1) << 52
    return struct.unpack("<d", struct.pack("<Q", m | (1 << 63 if neg else 0)))[0]


def test_fixed_point_accumulator_to_fp64():
    rng = random.Random(9)
    for _ in range(20000):
        b = rng.randint(0, 62)
        hi, s = rng.randint(-(1 << b), 1 << b), rng.randint(-900, 900)
        lo = rng.choice((0, 1, 0xFFFFFFFF, 0x80000000, rng.getrandbits(32), rng.getrandbits(8) << 24))
        exact = (Fraction(hi, 2**31) + Fraction(lo, 2**63)) * Fraction(2) ** s
        assert _fixed_scaled(hi, lo, s) == float(exact)


def test_group_sums_over_384_terms_stay_exact():
    worst = [384 * sum((128 if p == 0 else 64) * (128 if g == p else 64) for p in range(g + 1)) for g in range(8)]
    assert max(worst) < 2**24
    t = worst[2]
    for g in range(3, 8):
        t = t * 128 + worst[g]
    assert t < 2**59 and worst[0] * 128 + worst[1] < 2**30
