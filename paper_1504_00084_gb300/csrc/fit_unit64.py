"""Prints sdd_unit64.cuh: the tables of the FP64 path kernel's logarithm and sine / cosine.

log: u = 2^e m, m in [sqrt(1/2), sqrt(2)).  Entry i covers the m whose bits, less those of 1/2 + 2^-2.3,
start with i; its factor c is the reciprocal of the interval's middle rounded to 24 bits (1 next to
m = 1, so that ln u there is that of 1 + (m - 1) alone) and (hi, lo) is -ln c with hi a multiple of
2^-42.  Multiples e of ln 2 likewise.  sin, cos: the angles k 2 pi / 256 of the first quadrant, each
value as a rounded double and the rounded rest.
"""
import struct
from decimal import Decimal as D, getcontext

getcontext().prec = 60
OFF = 0x3FE6A00000000000  # bits of 0.70703125, just below sqrt(1/2)
N = 128


def dbl(bits):
    return struct.unpack("<d", struct.pack("<Q", bits))[0]


def split(x, unit=None):
    hi = float(x) if unit is None else float((x / unit).to_integral_value()) * float(unit)
    return hi, float(x - D(hi))


def trig(x):
    """sin x, cos x by their series."""
    s, c, t, n = D(0), D(0), D(1), 0
    while abs(t) > D(10) ** -58:
        if n % 2:
            s += t if n % 4 == 1 else -t
        else:
            c += t if n % 4 == 0 else -t
        n += 1
        t = t * x / n
    return s, c


def pi():
    """Machin's formula."""
    def arctan_inv(q):
        s, t, n = D(0), D(1) / q, 1
        while abs(t) > D(10) ** -58:
            s += t / n if n % 4 == 1 else -t / n
            t /= q * q
            n += 2
        return s
    return 4 * (4 * arctan_inv(5) - arctan_inv(239))


def log_entry(i):
    step = 1 << (52 - 7)
    a, b = OFF + i * step, OFF + (i + 1) * step
    # the interval straddles a power of two's exponent step only in value: its ends are doubles in
    # [0.707, 1.415)
    lo, hi = D(dbl(a)), D(dbl(b))
    if lo <= 1 <= hi or hi == 1:
        return 1.0, 0.0, 0.0
    c = struct.unpack("<f", struct.pack("<f", float(2 / (lo + hi))))[0]
    return (c, *split(-D(c).ln(), D(2) ** -42))


def main():
    P = pi()
    print("// Tables of the FP64 path kernel's logarithm and sine / cosine, printed by fit_unit64.py.")
    print("#pragma once\n")
    print("// factor, -ln factor (high part, rest), 0")
    print("alignas(32) __device__ const double kLog64[%d][4] = {" % N)
    for i in range(N):
        print("    {%s, %s, %s, 0.0}," % tuple(v.hex() for v in log_entry(i)))
    print("};\n// -e ln 2 (high part, rest), e = 0 .. 33")
    print("alignas(16) __device__ const double kLn2Times64[34][2] = {")
    hi, lo = split(D(2).ln(), D(2) ** -42)
    for e in range(34):
        h = -e * D(hi)
        print("    {%s, %s}," % (float(h).hex(), float(-e * D(2).ln() - h).hex()))
    print("};\n// sin, its rest, cos, its rest of k 2 pi / 256, k = 0 .. 63")
    print("alignas(32) __device__ const double kSinCos64[64][4] = {")
    for k in range(64):
        s, c = trig(2 * P * k / 256)
        print("    {%s, %s, %s, %s}," % tuple(v.hex() for v in split(s) + split(c)))
    print("};")
    step = 2 * P / 256
    print("// 2 pi, and 2 pi / 256 as a double and the rest")
    print("constexpr double kTwoPi64 = %s, kStep64 = %s, kStepRest64 = %s;" % (
        float(2 * P).hex(), float(step).hex(), float(step - D(float(step))).hex()))


if __name__ == "__main__":
    main()
