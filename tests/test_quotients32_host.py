"""The path kernel's paired FP32 quotients (quotients32 in sdd_mc.cu) on the host: its steps, emulated with
exactly rounded operations from every reciprocal estimate within 1 ulp (the hardware's bound), give the
correctly rounded a / d (no tolerance)."""
import random
from fractions import Fraction as F

import numpy as np
import pytest


def rn(x):
    """The float nearest to the Fraction x (even on ties); x in the normal range."""
    if x == 0:
        return F(0)
    s, x = (-1, -x) if x < 0 else (1, x)
    e = x.numerator.bit_length() - x.denominator.bit_length()
    e -= 0 if F(2) ** e <= x else 1
    u = F(2) ** (e - 23)
    n, r = divmod(x, u)
    n += 1 if r > u / 2 or (r == u / 2 and n % 2) else 0
    return s * n * u


def ru(x):
    """The least float not below x > 0."""
    r = rn(x)
    return r if r >= x else r + F(float(np.spacing(np.float32(r))))


def quotient(a, d, y):
    y = ru(y * rn(1 - d * y) + y)
    q = rn(a * y)
    for _ in range(2):
        q = rn(rn(a - q * d) * y + q)
    return q


def significands(rng, n):
    edge = [2 ** 23, 2 ** 23 + 1, 2 ** 24 - 1, 2 ** 24 - 2, 3 * 2 ** 22, 11863283]
    return edge + [rng.randrange(2 ** 23, 2 ** 24) for _ in range(n)]


@pytest.mark.parametrize("ea,ed", [(0, 0), (80 - 24, -20), (-60, 59), (-90, -20), (3, 8)])
def test_quotients_are_correctly_rounded(ea, ed):
    rng = random.Random(ea * 100 + ed)
    for md in significands(rng, 40):
        d = F(md) * F(2) ** (ed - 23)
        y0 = rn(1 / d)
        ulp = F(float(np.spacing(np.float32(y0))))
        for ma in significands(rng, 12):
            a = F(ma) * F(2) ** (ea - 23) * rng.choice([1, -1])
            want = rn(a / d)
            for k in (-1, 0, 1):
                assert quotient(a, d, y0 + k * ulp) == want
    assert quotient(F(0), F(3), rn(F(1, 3))) == 0
