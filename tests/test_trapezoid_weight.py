"""The weight of a fibre member (fibre_weight): the closed form of one coordinate
against the periodised sum it stands for, in exact rationals."""
from fractions import Fraction as F

import pytest


def _sum(t, q, eta, odd):
    """sum_n B(t / q + n) (-1)^(odd n), B the trapezoid of blend width eta."""
    u = F(0)
    for n in range(-3, 2):
        b = (F(1, 2) * (1 + eta) - abs(F(t, q) + n)) / eta
        u += min(max(b, F(0)), F(1)) * (-1 if odd * n % 2 else 1)
    return u


@pytest.mark.parametrize("eta", [F(1, 8), F(1, 3), F(3, 4), F(999, 1000)])
@pytest.mark.parametrize("q", [1, 2, 3, 8, 35, 243])
def test_closed_form(q, eta):
    for t in range(2 * q):
        x = 2 * abs(t - q) - q
        assert _sum(t, q, eta, 1) == min(max(F(x, 1) / (q * eta), F(-1)), F(1))
        assert _sum(t, q, eta, 0) == 1
