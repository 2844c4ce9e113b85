"""Integer tables of the fixed-point contractions (dg_fixed.cuh): every pair
(x, y) stands for the coefficient (x 2^31 + y) 2^(g - 62); checked against the
Gauss-Legendre values in double (whose own error is a few ulps), together
with the bounds that keep the 64-bit sums in range."""
import os
import re

import numpy as np
import pytest
from numpy.polynomial import legendre

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_08020_gb300", "csrc",
                   "dg_fixed.cuh")
TEXT = open(SRC).read()


def pairs(name, n):
    body = re.search(r"kFx%s%d\[\d+\] = \{(.*?)\};" % (name, n), TEXT, re.S).group(1)
    v = np.array([[int(x) for x in p] for p in re.findall(r"\{(-?\d+), (-?\d+)\}", body)], dtype=object)
    return v.reshape(-1, n, 2)


@pytest.mark.parametrize("n", range(2, 8))
def test_tables(n):
    x = legendre.leggauss(n)[0]
    A = np.array([np.sqrt((2 * p + 1) / 2) * legendre.Legendre.basis(p)(x) for p in range(n)])
    lag = [np.poly1d(np.poly(np.delete(x, r))) / np.prod(x[r] - np.delete(x, r)) for r in range(n)]
    D = np.array([np.polyder(p)(x) for p in lag])
    E = np.array([[p(y) for p in lag] for y in (-1.0, 1.0)])
    gA, gD = (int(re.search(r"FxTab<%d> \{\s+static constexpr int gA = (\d+), gD = (\d+);" % n, TEXT).group(k))
              for k in (1, 2))
    gE = int(re.search(r"kFxGE = (\d+);", TEXT).group(1))
    for name, ref, g, both in (("A", A, gA, True), ("D", D, gD, True), ("E", E, gE, False)):
        v = pairs(name, n)
        val = np.array([[float(p[0] * 2 ** 31 + p[1]) * 2.0 ** (g - 62) for p in row] for row in v])
        # the double reference: polynomials of degree < 7 in the monomial basis
        assert np.abs(val - ref).max() < 1e-12 * np.abs(ref).max()
        for rows in ([v, np.swapaxes(v, 0, 1)] if both else [v]):
            for row in rows:
                assert sum(abs(p[0] * 2 ** 31 + p[1]) for p in row) < 2 ** 62
                assert sum(abs(p[0]) * 2 ** 31 + abs(p[1]) * 2 ** 30 for p in row) < 2 ** 63
                assert all(-2 ** 30 <= p[1] < 2 ** 30 and -2 ** 31 <= p[0] < 2 ** 31 for p in row)
    # a lift adds a node's value and up to six face values
    ve = pairs("E", n)
    worst = max(sum(abs(ve[e, k, 0] * 2 ** 31 + ve[e, k, 1]) for e in (0, 1)) for k in range(n))
    assert 2 ** (62 - gE) + 3 * worst < 2 ** 62
