"""The FP64 kernels' arithmetic, operation by operation, against 60 decimal
digits: no less exact than the IEEE operations that it stands for."""
import math
from decimal import Decimal, getcontext

import numpy as np
import pytest

from paper_2409_09228_gb300 import fit

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU hosts too
    pytest.skip("needs a CUDA device", allow_module_level=True)

RCP, DIV, RSQRT, SQRT, TAN, SLOPE, ATAN = range(7)
getcontext().prec = 60
N = 20000


def _probe(op, x, y=None):
    x = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    y = torch.ones_like(x) if y is None else torch.from_numpy(np.ascontiguousarray(y)).cuda()
    out = torch.empty_like(x)
    fit.fit_probe_f64(op, x, y, out)
    return out.cpu().numpy()


def _worst(got, exact):
    """Largest error in units of the last place of the exact value."""
    return max(abs(Decimal(float(g)) - e) / Decimal(math.ulp(float(e))) for g, e in zip(got, exact))


def _numbers(seed, lo=-140, hi=140):
    """Random mantissas over the decades 10^lo..10^hi, some next to a power of two."""
    g = np.random.default_rng(seed)
    x = 10.0 ** g.uniform(lo, hi, N)
    near = np.ldexp(1.0, g.integers(-400, 400, N // 8)) * (1.0 + np.ldexp(g.integers(-8, 9, N // 8), -52))
    x[:N // 8] = near
    return x


# What IEEE operations reach, plus what is dropped: the coarse starts are good
# to 2^-20, so that e^3 = 2^-60 of the reciprocal's series and 5/16 (2^-19)^3
# of the reciprocal root's, below 0.02 units of the last place, are left out;
# the root's product x y rounds once more (half a unit).  Quotient and square
# root end with a step whose error is below 2^-70.
@pytest.mark.parametrize("op,bound", [(RCP, 0.52), (DIV, 0.5001), (RSQRT, 1.02), (SQRT, 0.5001)],
                         ids=["rcp", "div", "rsqrt", "sqrt"])
def test_units_of_the_last_place(op, bound):
    x, y = _numbers(139), _numbers(149) * np.where(np.arange(N) % 3 == 0, -1.0, 1.0)
    exact = {RCP: lambda a, b: 1 / a, DIV: lambda a, b: a / b, RSQRT: lambda a, b: 1 / a.sqrt(),
             SQRT: lambda a, b: a.sqrt()}[op]
    exact = [exact(Decimal(float(a)), Decimal(float(b))) for a, b in zip(x, y)]
    assert _worst(_probe(op, x, y), exact) <= bound


@pytest.mark.parametrize("op", [RCP, DIV, RSQRT, SQRT], ids=["rcp", "div", "rsqrt", "sqrt"])
def test_special_arguments_are_those_of_ieee(op):
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 1e-310, 2.0 ** -501, 2.0 ** -500, 2.0 ** 499,
                  2.0 ** 500, 1.7e308, 1.0, 4.0, 0.25])
    with np.errstate(all="ignore"):
        ref = {RCP: 1.0 / x, DIV: 3.0 / x, RSQRT: 1.0 / np.sqrt(x), SQRT: np.sqrt(x)}[op]
    got = _probe(DIV, np.full_like(x, 3.0), x) if op == DIV else _probe(op, x)
    np.testing.assert_array_equal(np.isnan(got), np.isnan(ref))
    ok = ~np.isnan(ref)
    np.testing.assert_allclose(got[ok], ref[ok], rtol=2.0 ** -52, atol=0.0)


# tan(theta) is one IEEE division's (half a unit); dh/dtheta = dz / cos^2 that
# of a product and a division (2^-53 of the value, one unit at most, and half).
@pytest.mark.parametrize("op,bound", [(TAN, 0.5001), (SLOPE, 1.5001)], ids=["tan", "slope"])
def test_plane_propagation_quotients(op, bound):
    g = np.random.default_rng(151)
    th = np.concatenate([g.uniform(0.01, np.pi - 0.01, N), np.pi / 2 + 10.0 ** g.uniform(-12, -1, 2000)])
    c = np.cos(th)
    x = np.sin(th) if op == TAN else g.uniform(-30.0, 30.0, c.size)
    exact = [Decimal(float(a)) / (Decimal(float(b)) if op == TAN else Decimal(float(b)) ** 2)
             for a, b in zip(x, c)]
    assert _worst(_probe(op, x, c), exact) <= bound


@pytest.mark.parametrize("op", [TAN, SLOPE], ids=["tan", "slope"])
def test_plane_propagation_at_the_ends_of_the_range(op):
    c = np.array([0.0, -0.0, 5e-324, 1e-200, 1e-160, 1.0, np.inf, np.nan])
    x = np.full_like(c, 1.5)
    with np.errstate(all="ignore"):
        ref = x / c if op == TAN else x / (c * c)
    np.testing.assert_allclose(_probe(op, x, c), ref, rtol=2.0 ** -50, atol=0.0)


def test_start_of_the_crossing():
    """atan(t) / t, both ranges of the series and their seam: half a unit for
    the last sum, an eighth for the terms left out (2^-56 below one), and the
    inner sums' roundings, at most 1/16 of a unit each way."""
    g = np.random.default_rng(157)
    t = np.concatenate([g.uniform(-0.25, 0.25, 4000), g.uniform(-0.0626, 0.0626, 4000),
                        10.0 ** g.uniform(-300, -2, 200),
                        [np.nextafter(0.25, 0), 0.0625, np.nextafter(0.0625, 0)]])
    t = t[np.abs(t) < 0.25]

    def ratio(a):
        v, term, total, k = -a * a, Decimal(1), Decimal(1), 1
        while abs(term) > Decimal(10) ** -40:
            term, k = term * v, k + 2
            total += term / k
        return total

    assert _worst(_probe(ATAN, t), [ratio(Decimal(float(a))) for a in t]) <= 0.75
