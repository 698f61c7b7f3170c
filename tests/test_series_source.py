"""The series of the particle kernels as their sources hold them: every
coefficient is the Taylor coefficient (FP32 literals: rounded to FP32, FP64
quotients: exactly), and the packed form's series truncate below 2^-28 at the
bounds under which it uses them (dxi <= 1/16, dt / r <= 1/40, nth >= 32)."""
import os
import re
from fractions import Fraction as Q
from math import factorial

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1407_1810_gb300", "csrc")
NUMBER = re.compile(r"(?<![\w.])(-?\d+\.\d*)f?(?:\s*/\s*(\d+\.\d*)f?)?")


def asin_c(k):  # t^(2k + 1)
    return Q(factorial(2 * k), 4 ** k * factorial(k) ** 2 * (2 * k + 1))


def binom(a, k):
    r = Q(1)
    for i in range(k):
        r *= (a - i) / Q(i + 1)
    return r


EXP = [Q(1, factorial(k)) for k in range(12)]
# function -> the numbers of its body, in the order they stand
SERIES = {
    ("tiles_two.cu", "exp_series"): [EXP[5], EXP[4], EXP[3], EXP[2], 1, 1],
    ("tiles_two.cu", "log1p_series"): [-Q(1, 6), Q(1, 5), -Q(1, 4), Q(1, 3), -Q(1, 2), 1],
    ("tiles_two.cu", "asin_series"): [asin_c(k) for k in (5, 4, 3, 2, 1)],
    ("tiles_two.cu", "asin_small"): [asin_c(2), asin_c(1)],
    ("tiles_two.cu", "cosm1_small"): [-binom(Q(1, 2), 3), binom(Q(1, 2), 2), -binom(Q(1, 2), 1)],
    ("tiles_two.cu", "inv_sqrt1p"): [binom(-Q(1, 2), k) for k in (6, 5, 4, 3, 2, 1, 0)],
    ("tiles_two.cu", "sin_cosm1_series"): [EXP[5], -EXP[3], 1, -EXP[6], EXP[4], -EXP[2]],
    ("tiles_one.cu", "exp_series"): [1, 1, EXP[2], EXP[3], EXP[4], EXP[5]],
    ("tiles_one.cu", "log1p_series"): [1, Q(1, 2), Q(1, 3), Q(1, 4), Q(1, 5), Q(1, 6)],
    ("tiles_one.cu", "atan_series"): [1, Q(1, 3), Q(1, 5), Q(1, 7)],
    ("tiles_one.cu", "sin_cosm1_series"): [EXP[5], EXP[3], 1, -Q(1, 2), 2 * EXP[6], 2 * EXP[4], 1],
    ("particles64.cu", "asin_series64"): [asin_c(k) for k in (8, 7, 6, 5, 4, 3, 2, 1)],
    ("particles64.cu", "exp_series64"): [EXP[k] for k in (8, 7, 6, 5, 4, 3, 2, 0, 0)],
    ("particles64.cu", "turn64"): [-EXP[9], EXP[7], -EXP[8], EXP[6], EXP[5], -EXP[3], EXP[4], -EXP[2]],
}


def body(file, name):
    s = open(os.path.join(CSRC, file)).read()
    m = re.search(r"\b%s\([^;{]*\)\s*\{(.*?)\n\}" % name, s, re.S)
    assert m, (file, name)
    return re.sub(r"//[^\n]*", "", m[1])


def numbers(text):
    return [Q(a) / Q(b or 1) if not a.endswith(".") or b else Q(a[:-1]) for a, b in NUMBER.findall(text)]


def is_coefficient(x, exact, fp32):
    return np.float32(float(x)) == np.float32(float(exact)) if fp32 else x == exact


@pytest.mark.parametrize("file,name", SERIES)
def test_coefficients(file, name):
    got, want = numbers(body(file, name)), SERIES[file, name]
    assert len(got) == len(want), got
    for x, e in zip(got, want):
        assert is_coefficient(x, Q(e), file != "particles64.cu"), (float(x), float(e))


def test_half_log1p_coefficients():
    got = [x for x in numbers(body("particles64.cu", "half_log1p64")) if x < Q(1, 2)]
    assert got == [Q(1, 11), Q(1, 9), Q(1, 7), Q(1, 5), Q(1, 3)]


def test_azimuth_coefficients_and_bound():
    """Three halvings take the angle from the x axis, at most pi / 2, to tan of
    at most pi / 16."""
    got = [x for x in numbers(body("tiles_two.cu", "azimuth")) if 0 < abs(x) < Q(1, 2) and abs(x) > Q(1, 12)]
    want = [-Q(1, 11), Q(1, 9), -Q(1, 7), Q(1, 5), -Q(1, 3)]
    assert len(got) == 5 and all(is_coefficient(x, e, True) for x, e in zip(got, want))
    t = np.tan(np.pi / 16)
    assert t ** 12 / 13 / (1 - t * t) < 2.0 ** -28
    a = np.linspace(1e-6, np.pi / 2, 20001)
    t = np.tan(a / 2)
    for _ in range(2):
        t = t / (1 + np.sqrt(1 + t * t))
    z = t * t
    p = -1 / 3 + z * (1 / 5 + z * (-1 / 7 + z * (1 / 9 - z / 11)))
    assert np.abs(8 * (t + t * z * p) / a - 1).max() < 2.0 ** -28


BOUND = Q(1, 2 ** 28)
EPS = Q(1, 40)                       # displacement of a step over r
SMAX = 2 * EPS + 3 * EPS ** 2        # |(r'/r)^2 - 1|


def test_packed_truncation_bounds():
    """First omitted terms, over 1 minus the ratio of the terms, relative to the
    leading one."""
    y = Q(1, 16)
    assert EXP[6] * y ** 6 / (1 - y) < BOUND * (1 - y)
    assert SMAX ** 6 / 7 / (1 - SMAX) < BOUND
    z = Q(1, 16)                     # azimuth below asin 1/4
    assert asin_c(6) * z ** 6 / (1 - z) < BOUND
    # the meridional turn: its sine is at most the displacement over r'
    t2 = (EPS / (1 - EPS)) ** 2
    assert asin_c(3) * t2 ** 3 / (1 - t2) < BOUND
    assert 2 * abs(binom(Q(1, 2), 4)) * t2 ** 3 / (1 - t2) < BOUND
    assert SMAX <= Q(52, 1000)
    assert abs(binom(-Q(1, 2), 7)) * SMAX ** 7 / (1 - SMAX) < BOUND
    b = Q(355, 113) / 32             # a cell of the linear theta map
    assert EXP[7] * b ** 6 < BOUND and 2 * EXP[8] * b ** 6 < BOUND
