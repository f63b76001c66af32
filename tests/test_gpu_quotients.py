"""The kernels' own division (accept factors and LU pivots) against exact quotients: both signs, mantissas
at and beside the powers of two, and exponents on both sides of the fall-back to the division.
"""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

afqmc = pytest.importorskip("paper_2506_09611_gb300.afqmc")

BOUND = Fraction(501, 1000)  # ulp of the result; a division has 1/2


def _mantissas(rng, n):
    """In [1, 2): the ends of the binade, 2^k above and below them, and random ones."""
    edge = [1.0 + 2.0 ** -k for k in range(1, 53)] + [2.0 - 2.0 ** -k for k in range(1, 53)] + [1.0]
    return np.concatenate([edge, 1.0 + rng.random(n)])


def _ulp_errors(got, num, den, bits, emin):
    """|got - num / den| in ulps of a result with `bits` significant bits, smallest exponent emin."""
    out = []
    for g, a, b in zip(got, num, den):
        exact = Fraction(float(a)) / Fraction(float(b))
        if exact == 0:
            out.append(Fraction(abs(float(g))))
            continue
        e = int(np.floor(np.log2(abs(float(exact)))))
        e += (abs(exact) >= Fraction(2) ** (e + 1)) - (abs(exact) < Fraction(2) ** e)
        out.append(abs(Fraction(float(g)) - exact) / Fraction(2) ** (max(e, emin) - bits + 1))
    return out


@pytest.mark.parametrize("ey", [-1000, -130, -101, -100, -99, -30, -1, 0, 1, 40, 99, 100, 101, 130, 1000])
def test_quotient_and_reciprocal_fp64(ey):
    rng = np.random.default_rng(abs(ey) + (ey < 0))
    m = _mantissas(rng, 600)
    y = np.ldexp(m * rng.choice([-1.0, 1.0], m.size), ey)
    x = np.ldexp(rng.permutation(m) * rng.choice([-1.0, 1.0], m.size), rng.integers(-8, 8, m.size))
    x[::50] = 0.0
    q, r, _ = afqmc.afqmc_debug_quotients(x, y)
    assert max(_ulp_errors(q, x, y, 53, -1022)) <= BOUND
    assert max(_ulp_errors(r, np.ones_like(y), y, 53, -1022)) <= BOUND


@pytest.mark.parametrize("ex,ey", [(-950, 50), (-950, -50), (950, 60), (-901, 3), (-900, 3), (900, 3), (901, 3)])
def test_quotient_fp64_far_numerators(ex, ey):
    rng = np.random.default_rng(1)
    m = _mantissas(rng, 200)
    x, y = np.ldexp(m, ex), np.ldexp(rng.permutation(m), ey)
    q, _, _ = afqmc.afqmc_debug_quotients(x, y)
    assert max(_ulp_errors(q, x, y, 53, -1022)) <= BOUND


def test_quotient_fp64_specials():
    x = np.array([1.0, -1.0, 0.0, np.inf, 1.0, 1.0, np.nan, 1.0, 5e-324, 1.0])
    y = np.array([0.0, 0.0, 0.0, 2.0, np.inf, -np.inf, 1.0, np.nan, 1.0, 5e-324])
    q, r, _ = afqmc.afqmc_debug_quotients(x, y)
    with np.errstate(all="ignore"):
        np.testing.assert_array_equal(q, x / y)
        np.testing.assert_array_equal(r, 1.0 / y)


@pytest.mark.parametrize("ey", [-100, -40, -1, 0, 1, 40, 100])
def test_quotient_fp32(ey):
    rng = np.random.default_rng(abs(ey) + (ey < 0))
    m = _mantissas(rng, 600).astype(np.float32).astype(np.float64)
    y = np.ldexp(np.minimum(m, 2.0 - 2.0 ** -23) * rng.choice([-1.0, 1.0], m.size), ey)
    x = np.ldexp(rng.permutation(m) * rng.choice([-1.0, 1.0], m.size), rng.integers(-8, 8, m.size))
    x[::50] = 0.0
    _, _, qf = afqmc.afqmc_debug_quotients(x, y)
    assert max(_ulp_errors(qf.astype(np.float64), x, y, 24, -126)) <= BOUND
