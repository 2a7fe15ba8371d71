"""recip_f64 and the negative powers of psi formed with it.

recip_f64: y + y (r + r^2) with y good to 2^-20 or better leaves r^3 < 2^-60, under 0.008 units of the last place, beside
the rounding of the last step (0.5) and 2^-53 |r|: 0.51 units over the whole range where neither x nor 1/x is
denormal; the limits at 0, infinity and NaN.

Powers: psi^2 enters psi^4 squared, so the worst error of psi^5, psi^6, psi^7 is 2 + 2, 3, 4 halves of a unit (relative to
2^-53, at most twice that in units of the last place of the result), and the reciprocal adds one half; the powers of the
correctly rounded 1/psi carry 5, 6, 7 times its half unit beside their own roundings, so both the largest and the mean
square error must come out no larger than theirs."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

L = np.longdouble


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from tests.native import load
    return load("powers")


def run(f, x, rows):
    xt = torch.from_numpy(x).cuda()
    out = torch.empty(rows * x.size, dtype=torch.float64, device="cuda")
    assert f(ctypes.c_void_p(xt.data_ptr()), ctypes.c_void_p(out.data_ptr()), x.size) == 0
    return out.cpu().numpy().reshape(rows, x.size)


def test_reciprocal(lib):
    rng = np.random.default_rng(0)
    m = np.concatenate([1 + rng.random(200000), [1.0, np.nextafter(2, 1), np.nextafter(1, 2), 1.5]])
    for e in (-1021, -1000, -500, -30, -1, 0, 1, 30, 500, 1000, 1020):
        x = np.ldexp(m, e) * rng.choice([-1.0, 1.0], m.size)
        y, exact = run(lib.recip, x, 1)[0], 1 / x.astype(L)
        ulps = np.abs(y - exact) / np.spacing(np.abs(exact).astype(np.float64))
        assert ulps.max() <= 0.51, (e, float(ulps.max()))
    edge = np.array([0.0, -0.0, np.inf, -np.inf, np.nan])
    with np.errstate(divide="ignore"):
        np.testing.assert_array_equal(run(lib.recip, edge, 1)[0], 1 / edge)


def test_powers_are_no_worse_than_those_of_a_rounded_reciprocal(lib):
    rng = np.random.default_rng(1)
    for lo, hi in ((0.5, 1.0), (0.99, 1.01), (1.0, 2.0), (1.0, 40.0)):
        psi = np.exp(rng.uniform(np.log(lo), np.log(hi), 300000))
        got = run(lib.powers, psi, 6)
        for r, k in enumerate((5, 6, 7)):
            exact = psi.astype(L) ** -k
            err = lambda v: np.abs(v - exact) / np.abs(exact) * 2.0 ** 53
            new, old = err(got[r]), err(got[3 + r])
            print(lo, hi, k, "largest %.2f %.2f, rms %.2f %.2f" % (new.max(), old.max(), np.sqrt((new ** 2).mean()), np.sqrt((old ** 2).mean())))
            assert new.max() <= k - 1 + 1 + 0.01, (lo, hi, k)
            assert new.max() <= old.max() and (new ** 2).mean() <= (old ** 2).mean(), (lo, hi, k)
