"""The ray clip divides by a known correctly rounded reciprocal (div_by in dvgo_internal.cuh: Markstein's two
corrections by the exact remainder).  The quotient must be the correctly rounded one: the same
operations, with exact fused multiply-adds formed from rationals, against IEEE division."""
from fractions import Fraction

import numpy as np


def fma(a, b, c):
    return float(Fraction(a) * Fraction(b) + Fraction(c))   # one rounding (int / int true division rounds correctly)


def div_by(a, b, y):
    q = a * y
    q = fma(fma(-q, b, a), y, q)
    return fma(fma(-q, b, a), y, q)


def test_div_by_is_correctly_rounded():
    g = np.random.default_rng(5)
    n = 4000
    mant = [g.integers(0, 2 ** 52, n), g.integers(0, 2 ** 23, n) << 29, 2 ** 52 - 1 - g.integers(0, 8, n)]
    for ma in mant:
        for mb in mant:
            a = np.ldexp(1.0 + ma / 2.0 ** 52, g.integers(-150, 3, n)) * g.choice([-1.0, 1.0], n)
            b = np.ldexp(1.0 + mb / 2.0 ** 52, g.integers(-270, 1, n)) * g.choice([-1.0, 1.0], n)
            for x, z in zip(a[:600].tolist(), b[:600].tolist()):
                assert div_by(x, z, 1.0 / z) == x / z, (x.hex(), z.hex())
    assert div_by(0.0, 0.3, 1.0 / 0.3) == 0.0
