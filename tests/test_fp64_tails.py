"""Square root and series with FP32 last terms of the FP64 particle step, their
operations replayed in numpy at the bounds of their arguments, against 50-digit
values.  Bounds: the FP32 part (conversion toward zero, rounded sums: 2^-22 of
it) is at most 2^-35 of the sum, so it adds less than 2^-57; the FP64 operations
round as they did, one ulp of the result (2^-52) in all."""
import math

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")
mp.mp.dps = 50
F, D = np.float32, np.float64


def low32(x):
    """FP64 -> FP32 toward zero with integer operations (|x| < 2)."""
    b = int(D(abs(x)).view(np.uint64))
    e = (b >> 32) - 0x38000000
    w = ((0 if e < 0x00100000 else e) << 3 | (b >> 29 & 7)) & 0xffffffff
    f = np.uint32(w).view(F)
    return -f if x < 0 else f


def high64(x):
    """Positive normal FP32 -> FP64 with integer operations."""
    b = int(F(x).view(np.uint32))
    return np.uint64(((b >> 3) + 0x38000000) << 32 | (b << 29 & 0xffffffff)).view(D)


def fma(a, b, c):
    return D(float(mp.mpf(float(a)) * mp.mpf(float(b)) + mp.mpf(float(c))))


def fmaf(a, b, c):
    return F(mp.mpf(float(a)) * mp.mpf(float(b)) + mp.mpf(float(c)))


def horner(p, z, cs):
    for c in cs:
        p = fma(p, z, c)
    return p


def asin(t):
    z, q = D(t) * D(t), F(6435.0 / 557056.0)
    for c in (143.0 / 10240.0, 231.0 / 13312.0, 63.0 / 2816.0):
        q = fmaf(q, low32(z), F(c))
    return fma(t * z, horner(high64(q), z, (35.0 / 1152.0, 5.0 / 112.0, 3.0 / 40.0, 1.0 / 6.0)), t)


def atanh(t):
    z = D(t) * D(t)
    p = high64(fmaf(F(1.0 / 11.0), low32(z), F(1.0 / 9.0)))
    return fma(t * z, horner(p, z, (1.0 / 7.0, 1.0 / 5.0, 1.0 / 3.0)), t)


def exp(x):
    y = low32(x)
    p = high64(fmaf(fmaf(F(1.0 / 40320.0), y, F(1.0 / 5040.0)), y, F(1.0 / 720.0)))
    return horner(p, x, (1.0 / 120.0, 1.0 / 24.0, 1.0 / 6.0, 0.5, 1.0, 1.0))


def sin(b):
    z = D(b) * D(b)
    p = high64(fmaf(F(-1.0 / 362880.0), low32(z), F(1.0 / 5040.0)))
    return fma(b * z, fma(fma(-p, z, 1.0 / 120.0), z, -1.0 / 6.0), b)


def cos(b):
    z = D(b) * D(b)
    q = high64(fmaf(F(-1.0 / 40320.0), low32(z), F(1.0 / 720.0)))
    return fma(fma(fma(-q, z, 1.0 / 24.0), z, -0.5), z, 1.0)


@pytest.mark.parametrize("form,value,bound", [
    (asin, mp.asin, 1 / 8), (atanh, mp.atanh, 1 / 31), (exp, mp.exp, 1 / 32),
    (sin, mp.sin, math.pi / 64), (cos, mp.cos, math.pi / 64)])
def test_fp32_tails(form, value, bound):
    g = np.random.default_rng(3)
    for x in [bound, bound / 2, bound / 1024, 1e-25, *(bound * (0.5 + 0.5 * g.random(40)))]:
        for s in (x, -x):
            ref = value(mp.mpf(float(s)))
            assert abs(mp.mpf(float(form(D(s)))) / ref - 1) <= mp.mpf(2) ** -52 + mp.mpf(2) ** -57
    if form is not atanh:
        assert form(D(0.0)) == (1.0 if form in (exp, cos) else 0.0)


def test_conversions():
    g = np.random.default_rng(4)
    for x in (g.random(200) + 1e-3) * 10.0 ** -g.integers(0, 30, 200):
        f = low32(D(x))
        assert 0 <= (x - float(f)) / x < 2.0 ** -23  # toward zero
        assert low32(D(-x)) == -f and high64(f) == D(f)
    assert abs(float(low32(D(1e-45)))) < 2.0 ** -126 and low32(D(0.0)) == 0


def test_square_root():
    """From approximations off by up to 2^-19: within one ulp."""
    g = np.random.default_rng(5)
    for x, e in zip(g.random(100) * 3 + 1, (g.random(100) * 2 - 1) * 2.0 ** -19):
        y = D((1 + e) / math.sqrt(x))
        r = D(x) * y
        t = fma(-r, r, x) * y
        v = fma(t, fma(0.375, t * y, 0.5), r)
        assert abs(mp.mpf(float(v)) / mp.sqrt(mp.mpf(float(x))) - 1) <= mp.mpf(2) ** -52
