"""The truncated series of the FP64 particle step, summed in exact rationals at
the bounds under which the step uses them: the first omitted term, which bounds
the rest, is below 2^-56 of the sum (an eighth of an FP64 ulp)."""
from fractions import Fraction as Q
from math import factorial


def _asin_coefficient(k):
    return Q(factorial(2 * k), 4 ** k * factorial(k) ** 2 * (2 * k + 1))


def test_asin_coefficients_and_bound():
    code = [Q(1, 6), Q(3, 40), Q(5, 112), Q(35, 1152), Q(63, 2816), Q(231, 13312), Q(143, 10240), Q(6435, 557056)]
    assert code == [_asin_coefficient(k) for k in range(1, 9)]
    # |t| < 1/8; the coefficients fall, so the rest is below the first omitted
    # term over 1 - t^2
    z = Q(1, 64)
    assert _asin_coefficient(9) * z ** 9 / (1 - z) < Q(1, 2 ** 56)


def test_half_log1p_bound():
    z = (Q(1, 16) / (2 - Q(1, 16))) ** 2  # (s / (2 + s))^2 at |s| = 1/16
    assert z ** 6 / 13 / (1 - z) < Q(1, 2 ** 56)


def test_exp_bound():
    x = Q(1, 32)  # half a cell at dxi = 1/16
    assert x ** 9 / factorial(9) / (1 - x) < Q(1, 2 ** 56)


def test_node_angle_turn_bound():
    b = Q(355, 113) / 64  # half a cell of pi / 32, pi from above
    assert b ** 11 / factorial(11) / b < Q(1, 2 ** 56)      # sin b / b
    assert b ** 10 / factorial(10) < Q(1, 2 ** 56)           # cos b - 1, against cos b


def test_third_order_steps_from_the_hardware_approximations():
    """Reciprocal and reciprocal square root from an approximation with
    relative error 2^-19 or less: the errors left by one step."""
    e = Q(1, 2 ** 19)
    for s in (e, -e):
        y = 1 + s  # x = 1
        d = 1 - y
        assert abs(y * (1 + d + d * d) - 1) < Q(1, 2 ** 56)
        d = 1 - y * y
        assert abs(y * (1 + d / 2 + 3 * d * d / 8) - 1) < Q(1, 2 ** 54)
