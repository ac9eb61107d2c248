"""The cut into nine-bit digits as ozaki.cu makes it, restated with Python integers: N = x 2^(9 D - e)
rounded to nearest even, in two's complement, plus 256 in every digit but the first, read as bit
fields. Checked: the digits give N back, they are at most 256, exact in bfloat16 (eight bits of
significand), and a prefix of s of them is within (1/2 + 1/511) 2^(-9 s) of the scaled x. Both forms
(6 and 8 digits), random numbers down to far below the row's largest, ties, carries through every
digit, rows of subnormal numbers and the ends of the exponent range."""
import math
import struct
from fractions import Fraction

import numpy as np
import pytest

BITS = 9


def parts(x):
    u = struct.unpack("<Q", struct.pack("<d", x))[0]
    xf, m = (u >> 52) & 0x7FF, u & ((1 << 52) - 1)
    return u >> 63, (m | (1 << 52), xf - 1075) if xf else (m, -1074)


def row_exponent(mx):
    """max |x| = m 2^e with m in [1/4, 1/2)"""
    return 0 if mx == 0 else 1 + math.frexp(mx)[1]


def digits(x, e, nd):
    sign, (m, ex) = parts(x)
    sh = BITS * nd - e + ex
    if sh >= 0:
        n = m << sh
    else:
        q, rem, half = m >> -sh, m & ((1 << -sh) - 1), 1 << (-sh - 1)
        n = q + (rem > half or (rem == half and q & 1))
    word = (-n if sign else n) & ((1 << 128) - 1)
    word = (word + sum(256 << (BITS * j) for j in range(nd - 1))) & ((1 << 128) - 1)
    out = []
    for s in range(1, nd + 1):
        f = word >> (BITS * (nd - s))
        if s > 1:
            out.append((f & 511) - 256)
        else:  # what remains, signed (the kernel keeps 32 bits of it)
            f &= (1 << 32) - 1
            out.append(f - (1 << 32) if f >> 31 else f)
    return out, (-n if sign else n)


def rows():
    rng = np.random.default_rng(0)
    yield rng.standard_normal(200)
    yield rng.standard_normal(200) * 2.0 ** rng.integers(-90, 1, 200)
    yield np.ldexp(1.0, rng.integers(-75, 1, 200))
    yield -np.ldexp(1.0 - 2.0 ** -53, rng.integers(-75, 1, 200))
    yield np.array([0.5 - 2.0 ** -54, 0.5, -0.5, 0.25] + [(257 + k) * 2.0 ** (-9 * s) for s in range(1, 9) for k in (-2, -1, -0.5, 0, 1)])
    yield np.array([(2 * k + 1) * 2.0 ** (-9 * s - 1) for s in range(1, 8) for k in range(-3, 4)] + [0.4])  # ties of every prefix
    yield np.ldexp(rng.integers(1, 1 << 40, 50).astype(float), -1074)
    yield np.array([5e-324, -5e-324, 1e-323])
    yield rng.standard_normal(50) * 2.0 ** 1020
    yield np.zeros(3)


@pytest.mark.parametrize("nd", [6, 8])
def test_digits(nd):
    for row in rows():
        e = row_exponent(float(np.abs(row).max()))
        for x in map(float, row):
            d, n = digits(x, e, nd)
            assert sum(v << (BITS * (nd - s)) for s, v in enumerate(d, 1)) == n
            assert all(abs(v) <= 256 for v in d)
            r = Fraction(x) * Fraction(2) ** -e
            assert abs(r) <= Fraction(1, 2)
            for s in range(1, nd + 1):
                prefix = sum(Fraction(v, 1 << (BITS * j)) for j, v in enumerate(d[:s], 1))
                assert abs(prefix - r) <= (Fraction(1, 2) + Fraction(1, 511)) / (1 << (BITS * s))
