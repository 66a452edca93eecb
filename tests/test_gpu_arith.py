"""Quotient, reciprocal, square root and reciprocal square root of the step
kernels (Newton-Raphson from the hardware's approximations) against correctly
rounded results. Before its last rounding the quotient is within 2^-90 of the
true one and the root within 2^-64 (relative), so a result other than the
correctly rounded one needs a true value that close to a tie: at most a 2^-11
share of the roots, practically no quotient, and then by one ulp. The
reciprocal square root carries the rounding of x y^2 besides its own: 1 ulp."""
import numpy as np
import pytest

from paper_2503_17608_gb300 import binding

pytestmark = pytest.mark.gpu

TINY, HUGE = 2.0 ** -510, 2.0 ** 510  # edges of the range taken without the operators


def operands(n):
    rng = np.random.default_rng(21)
    a = np.exp(rng.uniform(-30, 30, n)) * rng.choice([-1.0, 1.0], n)
    b = np.exp(rng.uniform(-60, 60, n)) * rng.choice([-1.0, 1.0], n)
    b[: n // 4] = 1.0 + rng.uniform(-1e-3, 1e-3, n // 4)  # divisors next to 1 and to powers of two
    b[n // 4 : n // 4 + 5] = [TINY, np.nextafter(TINY, 0), np.nextafter(HUGE, 0), HUGE, 1.0]
    return a, b


@pytest.mark.parametrize("fn", [0, 1])
def test_quotients_are_correctly_rounded(fn):
    a, b = operands(1_000_000)
    got = binding.debug_arith(fn, a, b)
    want = a / b if fn == 0 else 1.0 / b
    assert np.max(np.abs(got - want) / np.spacing(np.abs(want))) <= 1.0
    assert np.mean(got != want) <= 1e-5


def test_square_roots():
    x = np.abs(operands(1_000_000)[1])
    got, want = binding.debug_arith(2, x), np.sqrt(x)
    assert np.max(np.abs(got - want) / np.spacing(want)) <= 1.0
    assert np.mean(got != want) <= 2.0 ** -11
    inv = 1.0 / np.sqrt(x.astype(np.longdouble))
    err = np.abs(binding.debug_arith(3, x).astype(np.longdouble) - inv)
    assert float(np.max(err / np.spacing(inv.astype(np.float64)))) <= 1.0


@pytest.mark.parametrize("fn", [0, 1, 2, 3])
def test_other_operands_follow_the_operators(fn):
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 2.0 ** -1040, 1e308, -1e308, -1.0])
    a = np.ones_like(x) if fn < 2 else x
    with np.errstate(all="ignore"):
        want = {0: a / x, 1: 1.0 / x, 2: np.sqrt(x), 3: 1.0 / np.sqrt(x)}[fn]
        got = binding.debug_arith(fn, a, x)
        np.testing.assert_array_equal(np.isnan(got), np.isnan(want))
        ok = np.isfinite(want)
        np.testing.assert_array_equal(got[np.isinf(want)], want[np.isinf(want)])
        # CUDA's rsqrt is within 1 ulp, and 1 / np.sqrt too: two apart at most
        np.testing.assert_allclose(got[ok], want[ok], rtol=4.5e-16 if fn == 3 else 2.3e-16, atol=0)
