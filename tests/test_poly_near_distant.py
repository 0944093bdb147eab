"""The fits of poly_coeffs.h that near blocks and distant blocks evaluate, against
the closed form of two disjoint spheres: gn and hn up to GB_POLY_YNEAR, and the
coefficient lists GB_G2 .. GB_H3, each in FP32 Horner up to the largest (s/r)^2
its blocks may hold (GB_Y_G2 .. GB_Y_H3)."""
import math
import re

import numpy as np
import pytest

from test_poly_tables import CSRC, coeffs, horner32

HEADER = open(CSRC + "/poly_coeffs.h").read()


def _define(name):
    return re.search(r"#define %s (.*)" % name, HEADER).group(1)


def _list(name):
    return np.array([float(v.strip(" f")) for v in _define(name).strip("{}").split(",")], dtype=np.float32)


def _limit(name):
    return float(_define(name).rstrip("f"))


CASES = [("g", coeffs("gn"), _limit("GB_POLY_YNEAR")), ("h", coeffs("hn"), _limit("GB_POLY_YNEAR")),
         ("g", _list("GB_G3"), _limit("GB_Y_G3")), ("g", _list("GB_G2"), _limit("GB_Y_G2")),
         ("h", _list("GB_H3"), _limit("GB_Y_H3")), ("h", _list("GB_H2"), _limit("GB_Y_H2"))]


def _exact(f, y):
    """g(y) and h(y) from their Taylor series with every term positive:
    H = 1/(2r) [x/(1-x^2) - artanh x] = 1/2 s^3 r^-4 g(x^2), x = s/r, where the
    bracket is sum_k (1 - 1/(2k+1)) x^(2k+1), k >= 1; -r dH/dr = 1/2 s^3 r^-4 h
    takes 2k + 2 of each term's r^-(2k+2)."""
    s = [(1 - 1 / (2 * k + 1)) * (1 if f == "g" else 2 * k + 2) * y ** (k - 1) for k in range(80, 0, -1)]
    return np.sum(s, axis=0)


def test_series_is_the_closed_form():
    for x in (0.1, 0.3, 0.44):
        r = 1 / x
        H = lambda r: ((1 / r) / (1 - 1 / r ** 2) - math.atanh(1 / r)) / (2 * r)
        assert H(r) == pytest.approx(0.5 / r ** 4 * _exact("g", x * x), rel=1e-10)
        d = 1e-4 * r
        dH = (8 * (H(r + d) - H(r - d)) - (H(r + 2 * d) - H(r - 2 * d))) / (12 * d)
        assert -dH * r == pytest.approx(0.5 / r ** 4 * _exact("h", x * x), rel=1e-8)


@pytest.mark.parametrize("f,c,limit", CASES)
def test_fit_over_its_range(f, c, limit):
    """Within 2e-7: 6e-8 of the coefficients and two roundings of the last steps
    (the inner terms are small here), as the fits of the other ranges."""
    y = np.linspace(0.0, limit, 4001)
    y = np.minimum(y, np.float32(limit)).astype(np.float32)
    assert np.max(np.abs(horner32(c, y) / _exact(f, y.astype(np.float64)) - 1)) < 2e-7


def test_degrees_and_limits():
    assert [len(c) - 1 for _, c, _ in CASES[2:]] == [3, 2, 3, 2]
    assert _limit("GB_Y_G2") < _limit("GB_Y_G3") < _limit("GB_POLY_YFAR") < _limit("GB_POLY_YNEAR") < _limit("GB_POLY_YMAX")
    assert _limit("GB_Y_H2") < _limit("GB_Y_H3") < _limit("GB_POLY_YFAR")
