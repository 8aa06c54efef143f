"""The dot product that the FP64 kernels form on the integer and FP32 pipes (csrc/ddh_fixed.cuh), run on the
host against exact rational sums.

Bound: per component, 2^-52 P with P = sum of the absolute products in it.  (FP64 itself is bounded by
2 K 2^-53 P for K complex terms.  A component kept from the integer sum is rounded once, 2^-53 of at most
P, and the FP32 part adds 2^-72 to 2^-69 of the scale where P is 2^-16 of it or more, 2^-53 P at the most;
one formed in FP64 has random rounding errors, so it gets the FP64 bound.  The packed form's entries are
cut at 2^-64 of their scale, which makes 2^-64 to 2^-63 of the scale where P is 2^-10 of it or more, 2^-53 P,
one standard deviation: 2^-51 P.)"""
from fractions import Fraction

import numpy as np
import pytest


@pytest.fixture(scope="module", params=[False, True], ids=["split", "packed"])
def dot(request):
    from paper_1808_04713_gb300 import build as b
    b.build()
    from paper_1808_04713_gb300 import ddh

    def f(a, x, lanes):
        return ddh.fixed_dot(a, x, lanes, packed=request.param)
    f.tol = 2 if request.param else 1
    return f


def _exact(a, x):
    F = Fraction
    re = im = pr = pi = F(0)
    for u, v in zip(a, x):
        ar, ai, xr, xi = (F(float(t)) for t in (u.real, u.imag, v.real, v.imag))
        re += ar * xr - ai * xi
        im += ar * xi + ai * xr
        pr += abs(ar * xr) + abs(ai * xi)
        pi += abs(ar * xi) + abs(ai * xr)
    return (re, im), (pr, pi)


def _check(dot, a, x, lanes):
    y, fp64 = dot(a, x, lanes)
    ref, P = _exact(a, x)
    for c, got in enumerate((y.real, y.imag)):
        tol = P[c] * Fraction(max(1, len(a)) if fp64[c] else dot.tol, 2 ** 52)
        assert abs(Fraction(got) - ref[c]) <= tol, (c, fp64, got, float(ref[c]), float(P[c]))
    return y, fp64


def _rand(rng, K):
    return rng.standard_normal(K) + 1j * rng.standard_normal(K)


@pytest.mark.parametrize("K,lanes", [(0, 1), (1, 1), (2, 4), (76, 2), (124, 4), (128, 1), (255, 1), (256, 1), (300, 1),
                                     (1008, 32), (8192, 32)])
def test_random_and_one_sided_terms(dot, K, lanes):
    rng = np.random.default_rng(K)
    a, x = _rand(rng, K), _rand(rng, K)
    assert _check(dot, a, x, lanes)[1] == (False, False)
    # the largest limbs, all of one sign: no sum overflows, whatever the number of terms
    big = np.full(K, np.nextafter(2.0, 0.0))
    assert _check(dot, big * (1 - 1j), big * (1 + 1j), lanes)[1] == (False, False)
    assert _check(dot, -big * (1 + 0j), big * (1 + 1j), lanes)[1] == (False, False)


@pytest.mark.parametrize("g", [1e-4, 1e-8, 1e-12, 1e-17, 1e-30])
@pytest.mark.parametrize("K,lanes", [(76, 2), (300, 8)])
def test_graded_rows_and_vectors(dot, g, K, lanes):
    """Large entries of the row against small ones of the vector: what a scale shared by all entries loses."""
    rng = np.random.default_rng(1)
    t = g ** np.linspace(0.0, 1.0, K)
    a, x = _rand(rng, K), _rand(rng, K)
    _check(dot, a * t, x * t, lanes)
    _check(dot, a * t, x * t[::-1], lanes)
    # two regions: nothing of the vector's large part meets the row's
    half = np.where(np.arange(K) < K // 2, 1.0, g)
    _, fp64 = _check(dot, a * half, x * half[::-1], lanes)
    if g < 1e-4:                         # P is at most K g of the scale (at 1e-4: between the two forms' limits)
        assert fp64 == (True, True)
    # a small imaginary part of everything
    _check(dot, a.real * (1 + 0j), x.real + 1j * g * x.imag, lanes)
    _check(dot, a.real + 1j * g * a.imag, x, lanes)


def test_sums_that_cancel_stay(dot):
    rng = np.random.default_rng(2)
    a, x = _rand(rng, 64), _rand(rng, 64)
    a = np.concatenate([a, a * (1 + 1e-9)])
    x = np.concatenate([x, -x])
    assert _check(dot, a, x, 4)[1] == (False, False)


def test_zeros_are_exact_and_stay(dot):
    rng = np.random.default_rng(3)
    a, x = rng.standard_normal(80) * (1 + 0j), rng.standard_normal(80) * (1 + 0j)
    y, fp64 = _check(dot, a, x, 2)
    assert y.imag == 0.0 and fp64 == (False, False)
    assert dot(a, 0 * x, 2) == (0j, (False, False))
    assert dot(0 * a, x, 2) == (0j, (False, False))


@pytest.mark.parametrize("sa,sx", [(1e300, 1e-300), (1e-200, 1e150), (1e-150, 1e-150), (1e-290, 1.0), (1e-310, 1.0), (1e150, 1e150)])
def test_extreme_scales(dot, sa, sx):
    rng = np.random.default_rng(4)
    _check(dot, _rand(rng, 40) * sa, _rand(rng, 40) * sx, 2)


@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_non_finite_entries(dot, bad):
    rng = np.random.default_rng(5)
    a, x = _rand(rng, 40), _rand(rng, 40)
    x[7] = bad
    for u, v in ((a, x), (x, a)):
        y, fp64 = dot(u, v, 2)
        assert fp64 == (True, True) and not np.isfinite(y)
