"""The FP64 form's operations made from the hardware's estimates, each by itself
against the exact value (extended precision), over the exponent range.

Bounds, in u = 2^-53 relative (a rounding is at most u):
 1/x            the last FMA rounds once, the rest is third order: u
 a/x            (velocity recovery) rounded like a division: the error before its
                last rounding is some 2^-20 u, so it differs from the division only
                next to a tie, for about one value in 2^18
 sqrt(x)        the last rounding, and half of the rounding of x y: 1.5 u
 a/sqrt(x)      also the rounding of a y: 2.5 u
 each plus 0.1 u for the terms of higher order.
 fast speed     with D = G^2 - gamma p B_n^2 >= G^2 / 4: G u; G^2 and the product
                and D's own rounding 5 u G^2, so sqrt(D) 5 u G + 1.6 u sqrt(D);
                Q = G + sqrt(D) in [1.5, 2] G: at most 7.6 / 1.5 + 1 = 6.1 u; half
                of that and of Q rho's u, and the 2.6 u of the quotient: 6.2 u."""
import numpy as np
import pytest

from paper_2501_06717_gb300 import bats

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
L = np.longdouble


def _values(rng, n, lo, hi):
    return np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(lo, hi, n))


def _err(got, exact):
    return float(np.max(np.abs((got.astype(L) - exact) / exact))) / U


def test_reciprocal_roots_and_quotient():
    rng = np.random.default_rng(5)
    n = 400000
    x = _values(rng, n, -480, 480)
    a = _values(rng, n, -480, 480) * rng.choice([-1.0, 1.0], n)
    rcp, root, dsq, quo, _ = bats.bats_debug_fp64_ops(a, x)
    assert _err(rcp, 1 / x.astype(L)) <= 1.1
    assert _err(root, np.sqrt(x.astype(L))) <= 1.6
    assert _err(dsq, a.astype(L) / np.sqrt(x.astype(L))) <= 2.6
    assert _err(quo, a.astype(L) / x.astype(L)) <= 1.1
    assert np.mean(quo != a / x) <= 1e-4


def test_fast_speed():
    rng = np.random.default_rng(6)
    n = 400000
    rho = _values(rng, n, -200, 200)
    g = _values(rng, n, -200, 200)                  # gamma p / 2
    b = g * _values(rng, n, -6, 6)                  # B^2
    frac = rng.uniform(0.0, 1.0, n)
    G = g + b / 2
    c = np.minimum(frac * b, 0.74 * G * G / (2 * g))  # D >= G^2 / 4
    got = bats.bats_debug_fp64_ops(g, rho, b, c)[4]
    Gl = g.astype(L) + b.astype(L) / 2
    D = Gl * Gl - 2 * g.astype(L) * c.astype(L)
    assert _err(got, np.sqrt((Gl + np.sqrt(D)) / rho.astype(L))) <= 6.3
