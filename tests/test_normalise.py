"""Host-side check of the n-vector normalisation: for a squared length within a
few units in the last place of 1, the root found with integers and the
quotients (FP32: from a rounded reciprocal and two fused multiply-adds; FP64:
with integers) are the correctly rounded ones."""
from fractions import Fraction

import numpy as np
import pytest


@pytest.mark.parametrize("f,i,n", [(np.float32, np.int32, 1024), (np.float64, np.int64, 128)])
def test_root_near_one(f, i, n):
    one = int(np.array(1, f).view(i))
    d = np.arange(1 - n, n)
    assert (np.sqrt((one + d).astype(i).view(f)).view(i) == one + (d >> 1)).all()


def samples(f, rng, n=400):
    """Components in [-1, 1], with powers of two and their neighbours."""
    t = rng.uniform(-1, 1, n).astype(f)
    t[:60] = np.ldexp(f(1), -rng.integers(0, 20, 60)).astype(f)
    t[20:40] = np.nextafter(t[20:40], f(2))
    t[40:60] = np.nextafter(t[40:60], f(0))
    return t


def round32(x):
    """A Fraction rounded to the nearest float32, ties to even."""
    if x == 0:
        return np.float32(0)
    e = 0
    a = abs(x)
    while a * Fraction(2) ** -e >= 1 << 24:
        e += 1
    while a * Fraction(2) ** -e < 1 << 23:
        e -= 1
    m = a * Fraction(2) ** -e
    k = m.numerator // m.denominator
    rest = m - k
    k += rest > Fraction(1, 2) or (rest == Fraction(1, 2) and k & 1)
    return np.float32(np.ldexp(float(k), e) * (1 if x > 0 else -1))


def test_fp32_quotients():
    rng = np.random.default_rng(4)
    for h in (-512, -130, -7, -3, -2, -1, 1, 2, 3, 9, 127, 511):
        s = np.array(0x3F800000 + h, np.int32).view(np.float32)
        r = np.float32(1) / s
        fs, fr = Fraction(float(s)), Fraction(float(r))
        for t in samples(np.float32, rng):
            ft = Fraction(float(t))
            g = round32(ft - (fs - 1) * ft)  # one fma
            fg = Fraction(float(g))
            res = ft - fs * fg
            assert Fraction(float(round32(res))) == res  # exact in one fma
            assert round32(res * fr + fg) == t / s


def test_fp64_quotients():
    rng = np.random.default_rng(5)
    one, field = 0x3FF0000000000000, (1 << 52) - 1
    for h in range(-64, 64):
        if h == 0:
            continue
        s = np.array(one + h, np.int64).view(np.float64)
        t = samples(np.float64, rng)
        m, sh = abs(h), 52 if h > 0 else 53
        D = (1 << sh) + h
        taken = 0
        for x, want in zip(t, t / s):
            b = int(x.view(np.uint64))
            mant = b & field
            n = (mant | (1 << 52)) * m
            assert n < 1 << 59
            k = (n + (1 << (sh - 1))) >> sh
            r2 = 2 * (n - k * D)
            k += -(r2 < -D) if h > 0 else (r2 > D)
            to = mant - k if h > 0 else mant + k
            if 0 <= to <= field:  # else the kernel divides
                taken += 1
                assert (b - k if h > 0 else b + k) == int(want.view(np.uint64))
        assert taken > 330
