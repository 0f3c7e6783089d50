"""The kernels' quotients, roots and reciprocals from the hardware's approximations and one
correction (adjoint.cu quot and root, solver.cuh rcp_newton), restated in exact arithmetic:
for every approximation within the error CUDA's PTX manual states (rcp.approx 1 ulp,
rsqrt.approx 2^-22.9 relative) the corrected value is the correctly rounded one, up to a
share of cases next to a rounding boundary, and never further off than one unit in the last
place.  The range for which this holds is the one the kernels guard."""
import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1904_02833_gb300", "csrc")
F, D = np.float32, np.float64


def fma(a, b, c):
    """a b + c rounded once (the product is exact in 64 bits; the sum's own rounding there
    matters only within 2^-29 of a 32-bit rounding boundary)."""
    return (D(a) * D(b) + D(c)).astype(F)


def operands(rng, n, lo, hi):
    return np.ldexp(rng.uniform(1, 2, n), rng.integers(lo, hi, n)).astype(F)


def off(x, exact):
    """Distance from the correctly rounded value in units of the last place."""
    r = exact.astype(F)
    return np.abs(D(x) - D(r)) / D(np.spacing(np.abs(r)))


@pytest.mark.parametrize("ulps", [-1, 0, 1])
@pytest.mark.parametrize("size", [2.0 ** -21, 2.0 ** -6, 1.0, 2.0 ** 20.4])
def test_shared_reciprocal_quotients_of_a_segment(ulps, size):
    """The quotients of a segment's derivatives, with the segment at the ends of the guarded
    range and between (the remainder a - b q must not underflow, which the numerators of
    such segments see to)."""
    rng = np.random.default_rng(9)
    n = 100000
    ang, tilt = rng.uniform(0.05, 1.5, n), rng.uniform(0.05, 1.2, n)
    rho = size * rng.uniform(1, 1.05, n)
    x, y, z = (v.astype(F) for v in (rho * np.cos(ang), rho * np.sin(ang), np.minimum(rho * np.tan(tilt), 2.0 ** 20.4)))
    with np.errstate(all="raise"):
        xx, yy = x * x, y * y
        rho2 = xx + yy
        rho, r2 = np.sqrt(rho2), rho2 + z * z
        assert rho2.min() >= 2.0 ** -42 and r2.max() <= 2.0 ** 42
        r4, q = r2 * r2, rho * r2
        dq = F(2) * rho + r2 / rho
        pairs = [(x, np.sqrt(r2)), (y, rho2), (z * x, q), (rho, r2), (F(2) * x * y, rho2 * rho2), (x, q),
                 (z * x * x * dq, q * q), (F(2) * z * z * x, rho * r4), (F(2) * rho * z, r4), (r2, rho)]
        for a, b in pairs:
            rb = (1 / D(b)).astype(F)
            rb = rb + F(ulps) * np.spacing(rb)
            p = (a * rb).astype(F)
            e = off(fma(fma(-b, p, a), rb, p), D(a) / D(b))
            assert e.max() <= 1 and (e > 0).mean() <= 1e-4


@pytest.mark.parametrize("rel", [-2 ** -22.9, 0.0, 2 ** -22.9])
def test_root_from_the_approximate_reciprocal_root(rel):
    rng = np.random.default_rng(7)
    x = operands(rng, 400000, -42, 42)
    y = (1 / np.sqrt(D(x)) * (1 + rel)).astype(F)
    s = (x * y).astype(F)
    r = fma(fma(-s, s, x), (F(0.5) * y).astype(F), s)
    e = off(r, np.sqrt(D(x)))
    assert e.max() <= 1 and (e > 0).mean() <= 1e-4


@pytest.mark.parametrize("ulps", [-1, 0, 1])
def test_reciprocal_of_steep_tangents(ulps):
    rng = np.random.default_rng(8)
    a = np.concatenate([operands(rng, 400000, 0, 12), operands(rng, 4000, 100, 126)])
    y = (1 / D(a)).astype(F) + F(ulps) * np.spacing((1 / D(a)).astype(F))
    e = off(fma(fma(-a, y, np.ones_like(a)), y, y), 1 / D(a))
    assert e.max() <= 1 and (e > 0).mean() <= 1e-4


def test_guarded_range_keeps_every_divisor_normal():
    src = open(os.path.join(CSRC, "adjoint.cu")).read()
    lo, hi = (float(v) for v in re.search(r"e\.lo >= ([\d.e+-]+)f && e\.hi <= ([\d.e+-]+)f", src).groups())
    lo, hi = D(F(lo)), D(F(hi))  # of rho^2 and r^2, rho <= r
    for rho2 in (lo, hi):
        for r2 in (rho2, hi):
            rho, r4 = np.sqrt(rho2), r2 * r2
            for b in (rho2, rho2 * rho2, rho, rho * r2, rho2 * r4, rho * r4, r2, r4, np.sqrt(r2)):
                assert 2.0 ** -126 <= b <= 2.0 ** 126
    cap = float(re.search(r"fminf\(D \+ at, ([\d.e+]+)f\)", src).group(1))
    assert D(F(cap)) == 2.0 ** 126
