"""The float32 merged mean's division step (sample.cuh, mean_of for float), restated in exact rational
arithmetic with one rounding per operation: the quotient it returns is the correctly rounded one, ties
included.  This is the arithmetic alone, for divisors that are floats; test_gpu_mean_rounding.py holds the kernel's
output to it."""
from fractions import Fraction

import numpy as np


def rn(v: Fraction) -> Fraction:
    """v rounded to float32, ties to even (normal range)."""
    if v == 0:
        return v
    e = 0
    a = abs(v)
    while a >= 2 ** (e + 1):
        e += 1
    while a < Fraction(2) ** e:
        e -= 1
    ulp = Fraction(2) ** (e - 23)
    n = v / ulp
    f = n.numerator // n.denominator
    r = n - f
    if r > Fraction(1, 2) or (r == Fraction(1, 2) and f % 2):
        f += 1
    return f * ulp


def two_sum(a, b):
    s = rn(a + b)
    return s, (a + b) - s


def mean_of(nh, nl, den):
    """(num.hi, num.lo) / den, den a float with lo part 0; the reciprocal is given to float32."""
    inv = rn(Fraction(1) / den)
    q1 = rn(nh * inv)
    ph = rn(q1 * den)
    pl = q1 * den - ph
    ah, al = two_sum(rn(nh - ph), -pl)
    bh, bl = two_sum(ah, nl)
    r = rn(bh + rn(al + bl))
    q2 = rn(r * inv)
    q2 = rn(q2 + rn(r - q2 * den) * inv)
    return rn(q1 + q2)


def f32(rng, n):
    return [Fraction(float(v)) for v in (rng.standard_normal(n) * 2.0 ** rng.integers(-6, 7, n)).astype(np.float32)]


def test_quotient_is_correctly_rounded():
    rng = np.random.default_rng(0)
    for den in (2, 3, 5, 6, 7, 11, 12, 13, 63, 100, 197):
        den = Fraction(den)
        for x, y in zip(f32(rng, 60), f32(rng, 60)):
            s = x * (den - 1) + y   # a size-weighted sum, as high and low parts
            nh = rn(s)
            nl = rn(s - nh)
            assert mean_of(nh, nl, den) == rn((nh + nl) / den)


def test_exact_ties_go_to_even():
    rng = np.random.default_rng(1)
    for den in (3, 5, 6, 7, 11, 13):
        den = Fraction(den)
        for x in f32(rng, 60):
            m = rn(x)
            e = 0
            while abs(m) >= Fraction(2) ** (e + 1):
                e += 1
            while abs(m) < Fraction(2) ** e:
                e -= 1
            mid = m + Fraction(2) ** (e - 24)   # halfway to the next float
            s = mid * den
            nh = rn(s)
            nl = s - nh
            assert rn(nl) == nl
            assert mean_of(nh, nl, den) == rn(mid)
