"""The FP64 path kernel's quotients64 and sqrt_four64 (sdd_mc.cu) over the whole range that their own tests accept:
the steps, emulated with exactly rounded operations from every hardware estimate within 1 ulp, subnormal ones
flushed to zero as the instructions do, stay within 0.51 ulp of the exact result (half an ulp of the last rounding, and
what the reciprocal's error, 2^-50 at most, leaves of the residual)."""
import math
import os
import random
import re
import struct
from fractions import Fraction as F

import numpy as np
import pytest

SRC = open(os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1504_00084_gb300", "csrc",
                        "sdd_mc.cu")).read()


def body(name):
    i = SRC.index(name + "(double")
    return SRC[i:SRC.index("\n}\n", i)]


def hi(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0] >> 32


def from_words(h, l):
    return struct.unpack("<d", struct.pack("<Q", ((h & 0xFFFFFFFF) << 32) | (l & 0xFFFFFFFF)))[0]


def fma(a, b, c):
    v = F(a) * F(b) + F(c)
    try:
        return float(v)
    except OverflowError:
        return math.inf if v > 0 else -math.inf


def upper_float(d):
    return np.uint32((((hi(d) << 3) | ((struct.unpack("<Q", struct.pack("<d", d))[0] & 0xFFFFFFFF) >> 29)) + 0x40000000)
                     & 0xFFFFFFFF).view(np.float32)


def estimates(v):
    """Bits of the floats within 1 ulp of v > 0, subnormal ones flushed."""
    f = np.float32(v)
    for g in (f, np.nextafter(f, np.float32(0)), np.nextafter(f, np.float32(np.inf))):
        yield 0 if g < np.float32(2.0 ** -126) else int(np.float32(g).view(np.uint32))


def accepted_range(name):
    lo, n = re.search(r"hi - (0x[0-9A-F]+)\) >= (0x[0-9A-F]+)u", body(name)).groups()
    return int(lo, 16), int(lo, 16) + int(n, 16)


def ends(name, rng):
    """Arguments at both ends of the accepted range, next to powers of two and spread over it."""
    lo, end = accepted_range(name)
    e0, e1 = (lo >> 20) - 1023, (end >> 20) - 1023  # [2^e0, 2^e1)
    assert lo & 0xFFFFF == 0 and end & 0xFFFFF == 0
    for e in [e0, e0 + 1, e0 + 2, -1, 0, 1, e1 - 3, e1 - 2, e1 - 1] + [rng.randrange(e0, e1) for _ in range(10)]:
        for m in [1.0, 1.0 + 2.0 ** -52, 2.0 - 2.0 ** -52, 2.0 - 2.0 ** -24, 1.75] + [rng.uniform(1, 2) for _ in range(6)]:
            yield math.ldexp(m, e)


def ulps(got, want):
    return abs(F(got) - want) / F(math.ulp(got)) if math.isfinite(got) else math.inf


def test_quotients_over_the_accepted_range():
    rng = random.Random(1)
    cut = re.search(r"most >= (0x[0-9A-F]+)u", body("quotients64"))
    top = (int(cut.group(1), 16) >> 20) - 1023 if cut else 1024  # numerators below 2^top
    for d in ends("quotients64", rng):
        for ea in (0, -300, 300, top - 1, rng.randrange(-800, top)):
            a = math.ldexp(rng.uniform(1, 2), ea) * rng.choice([1, -1])
            exact = F(a) / F(d)
            if not cut and abs(exact) >= F(2) ** 1024:
                exact = None  # an infinity, which the steps have to give
            for yb in estimates(1.0 / float(upper_float(d))):
                y0 = from_words((yb >> 3) + 0x38000000, yb << 29)
                y1 = fma(y0, fma(-d, y0, 1.0), y0)
                y2 = fma(y1, fma(-d, y1, 1.0), y1)
                u = fma(a, y2, 0.0)
                assert math.isfinite(u), (a, d)
                q = fma(fma(-u, d, a), y2, u)
                assert exact is not None and ulps(q, exact) <= F(51, 100), (a, d, q)


def test_roots_over_the_accepted_range():
    rng = random.Random(2)
    for a in ends("sqrt_four64", rng):
        a2 = 4.0 * a
        s = F(math.isqrt(int(F(a2) * F(2) ** 400)), 2 ** 200)  # to 2^-200
        for yb in estimates(1.0 / math.sqrt(float(upper_float(a2)))):
            yh = (yb >> 3) + 0x38000000
            y0, h0 = from_words(yh, yb << 29), from_words(yh - 0x00100000, yb << 29)
            t = a2 * y0
            e = fma(-t, h0, 0.5)
            g, h = fma(t, e, t), fma(h0, e, h0)
            assert ulps(fma(fma(-g, g, a2), h, g), s) <= F(51, 100), a


@pytest.mark.parametrize("name", ["quotients64", "sqrt_four64"])
def test_range_is_where_the_seed_is_normal(name):
    lo, end = accepted_range(name)
    assert 0x38100000 <= lo < end <= 0x47F00000  # upper_float: [2^-126, 2^128)
