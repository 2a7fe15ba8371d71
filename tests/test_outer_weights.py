"""The fused residual's weights against 1/h^2, 1/(h h') and 1/h: spacings that are equal, that (hi - lo) / n left one or
two units of the last place apart, and unequal ones.

Bound, in units of 2^-53: a weight is one rounded constant (1 unit); equal spacings share one weight, formed from
the mean of the smallest and the largest, which one unit of the last place (2 units) apart lie 1 unit from it
each, 2 in 1/h^2; so 3 units, as many as a rounded 1 / (h h) times a rounded stencil weight has.  Unequal spacings
share the smallest spacing's weight by ratios in 64-bit fixed point, so there the bound is 3 units of that weight."""
import ctypes
import math

import pytest

from tests.native import load


@pytest.fixture(scope="module")
def errors():
    f = load("outer_weights").outer_weight_errors

    def run(h, order):
        e = (ctypes.c_double * 21)()
        return f((ctypes.c_double * 3)(*h), order, e), list(e)
    return run


def up(x, n):
    for _ in range(n):
        x = math.nextafter(x, math.inf)
    return x


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("base", [1.0, 0.25, 0.3, 1.9999999, 7.3e-5, 1e6])
@pytest.mark.parametrize("apart", [(0, 0, 0), (0, 1, 0), (1, 0, 1), (0, 2, 1), (3, 0, 0)])
def test_nearly_equal_spacings(errors, base, apart, order):
    iso, e = errors([up(base, n) for n in apart], order)
    assert iso == (max(apart) <= 1)
    assert max(e) <= 3.0, e


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("h", [(1.0, 1.25, 0.75), (0.33, 0.4, 0.508), (0.1, 0.1, 3.0), (2.0, 0.01, 0.3)])
def test_unequal_spacings(errors, h, order):
    iso, e = errors(h, order)
    assert not iso
    share = [min(h) / x for x in h]
    assert all(e[r + a] * share[a] ** 2 <= 3.0 for r in (0, 3, 6, 9) for a in range(3)), e
    assert all(x <= 3.0 for x in e[12:18]), e
    assert all(e[18 + a] * share[a] <= 3.0 for a in range(3)), e
