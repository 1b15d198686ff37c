"""The FP64 path kernel's logarithm and sine / cosine (sdd_mc.cu) on the host: the committed tables are
what fit_unit64.py prints, and the kernels' steps, emulated with exactly rounded operations, stay
within 0.51 ulp (logarithm) and 1.5 ulp (sine, cosine, whose worst is next to their zeros) of
50-digit arithmetic."""
import contextlib
import io
import math
import os
import random
import re
import struct
import sys
from decimal import Decimal as D
from fractions import Fraction as F

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1504_00084_gb300", "csrc")
sys.path.insert(0, CSRC)
import fit_unit64 as G  # noqa: E402

HEADER = open(os.path.join(CSRC, "sdd_unit64.cuh")).read()


def table(name):
    i = HEADER.index("{", HEADER.index(name + "["))
    return [[float.fromhex(v.strip()) for v in r.split(",")]
            for r in re.findall(r"\{([^{}]+)\}", HEADER[i + 1:HEADER.index("};", i)])]


def constant(name):
    return float.fromhex(re.search(name + r" = ([^,;]+)", HEADER).group(1))


def fma(a, b, c):
    return float(F(a) * F(b) + F(c))


def bits(x):
    return struct.unpack("<q", struct.pack("<d", x))[0]


def words(n):
    rng = random.Random(n)
    w = [0, 1, 2, 2 ** 32 - 1, 2 ** 32 - 2, 2 ** 31, 2 ** 31 - 1, 2 ** 30, 3 * 2 ** 30 - 1]
    w += [rng.randrange(2 ** 32) for _ in range(n)]
    for k in range(1, 32):  # every binade of u and of 1 - u, and both sides of the quadrants
        w += [rng.randrange(2 ** k), 2 ** 32 - 1 - rng.randrange(2 ** k)]
        w += [(q * 2 ** 30 + rng.randrange(-2 ** k, 2 ** k)) % 2 ** 32 for q in range(4)]
    return w


def ulps(got, want):
    return abs(float((D(got) - want) / D(math.ulp(got))))


def test_tables_are_what_the_generator_prints():
    out = io.StringIO()
    with contextlib.redirect_stdout(out):
        G.main()
    assert out.getvalue() == HEADER


def test_logarithm():
    L, E = table("kLog64"), table("kLn2Times64")
    for w in words(400):
        u = (w + 0.5) * 2.0 ** -32
        tmp = (bits(u) >> 32) - 0x3FE6A000
        i, e = (tmp >> 13) & 127, tmp >> 20
        m = math.ldexp(u, -e)
        c, h, l, _ = L[i]
        eh, el = E[-e]
        r = fma(m, c, -1.0)
        assert F(r) == F(m) * F(c) - 1 and F(eh + h) == F(eh) + F(h)
        hi = eh + h
        s = hi + r
        lo = ((hi - s) + r) + (el + l)
        p = fma(r, 1.0 / 7, -1.0 / 6)
        for q in (1.0 / 5, -1.0 / 4, 1.0 / 3, -1.0 / 2):
            p = fma(p, r, q)
        assert ulps(s + fma(r * r, p, lo), D(u).ln()) <= 0.51


@pytest.mark.parametrize("n", [300])
def test_sine_and_cosine(n):
    T = table("kSinCos64")
    two_pi, step, rest = constant("kTwoPi64"), constant("kStep64"), constant("kStepRest64")
    for w in words(n):
        t = two_pi * ((w + 0.5) * 2.0 ** -32)
        k = ((w >> 23) + 1) >> 1
        y = fma(-float(k), step, t)
        assert F(y) == F(t) - k * F(step)
        y = fma(-float(k), rest, y)
        y2 = y * y
        p = fma(fma(y2, -1.0 / 5040, 1.0 / 120), y2, -1.0 / 6)
        sy = fma(p * y2, y, y)
        cm = fma(fma(y2, -1.0 / 720, 1.0 / 24), y2, -0.5) * y2
        S, Sr, C, Cr = T[k & 63]
        s = S + fma(C, sy, fma(S, cm, Sr))
        c = C + fma(-S, sy, fma(C, cm, Cr))
        q = k >> 6
        if q & 1:
            s, c = c, s
        s, c = (-s if q & 2 else s), (-c if (q + 1) & 2 else c)
        es, ec = G.trig(D(t))
        assert ulps(s, es) <= 1.5 and ulps(c, ec) <= 1.5
