"""Integer tables of the contractions to the last unit, and the bounds that
keep their 64-bit sums from overflowing."""
import ctypes
import os
import re

import pytest

from fixed_host import CSRC, fx  # noqa: F401

TEXT = open(os.path.join(CSRC, "dg_fixed.cuh")).read()


def body(name, n):
    return re.search(r"kFx%s%d\[\d+\] = \{(.*?)\};" % (name, n), TEXT, re.S).group(1)


def pairs(name, n):
    return [tuple(map(int, p)) for p in re.findall(r"\{(-?\d+), (-?\d+)\}", body(name, n))]


@pytest.mark.parametrize("n", range(2, 8))
def test_coefficients_to_the_last_unit(n):
    mp = pytest.importorskip("mpmath")
    with mp.workdps(50):
        p0, p1 = [mp.mpf(1)], [mp.mpf(0), mp.mpf(1)]           # P_n's coefficients by the recurrence
        for k in range(2, n + 1):
            up = [mp.mpf(0)] + [(2 * k - 1) * c / k for c in p1]
            p0, p1 = p1, [c - (mp.mpf(k - 1) / k * p0[i] if i < len(p0) else 0) for i, c in enumerate(up)]
        x = sorted(mp.re(v) for v in mp.polyroots(p1[::-1], maxsteps=200, extraprec=200))
        assert len(x) == n and max(abs(mp.polyval(p1[::-1], v)) for v in x) < mp.mpf(10) ** -45
        x = [(a - b) / 2 for a, b in zip(x, x[::-1])]

        def lagrange(m, y):
            return mp.fprod((y - x[k]) / (x[m] - x[k]) for k in range(n) if k != m)

        def slope(m, i):
            if m == i:
                return mp.fsum(1 / (x[m] - x[k]) for k in range(n) if k != m)
            return mp.fprod(x[i] - x[k] for k in range(n) if k not in (m, i)) / mp.fprod(x[m] - x[k] for k in range(n) if k != m)
        A = [mp.sqrt(mp.mpf(2 * p + 1) / 2) * mp.legendre(p, x[i]) for p in range(n) for i in range(n)]
        D = [slope(r, i) for r in range(n) for i in range(n)]
        E = [lagrange(m, y) for y in (-1, 1) for m in range(n)]
        gA, gD = (int(re.search(r"FxTab<%d> \{\s+static constexpr int gA = (\d+), gD = (\d+);" % n, TEXT).group(k)) for k in (1, 2))
        gE = int(re.search(r"kFxGE = (\d+);", TEXT).group(1))
        for name, ref, g in (("A", A, gA), ("D", D, gD), ("E", E, gE)):
            got = pairs(name, n)
            assert len(got) == len(ref)
            for (u, v), c in zip(got, ref):
                assert abs((u * 2 ** 31 + v) - c * mp.mpf(2) ** (62 - g)) <= 1
        # 2^30 and the mean of the products that a derivative sum leaves out
        S = [int(v) for v in re.findall(r"-?\d+", body("S", n))]
        for r in range(n):
            assert abs(S[r] - (2 ** 30 + sum(v for _, v in pairs("D", n)[r * n:(r + 1) * n]) / 2)) <= 1


@pytest.mark.parametrize("n", range(2, 8))
@pytest.mark.parametrize("etype", range(4))
def test_sums_fit(fx, n, etype):  # noqa: F811
    fx.t_bounds.restype = ctypes.c_double
    assert fx.t_bounds(n, etype) < 1
