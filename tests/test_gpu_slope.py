"""Half limited slopes of the FP64 flux kernels against their definition in IEEE arithmetic: minmod and the
monotonised central limiter to the bit (halvings are exact, or rounded once below the normal range),
van Leer a b / (a + b) within one ulp of the rounded product over the rounded sum; from subnormal
differences to sums beyond the range, and an infinite difference beside a finite one."""
import numpy as np
import pytest

from paper_2501_15923_gb300 import inputs as I

from .test_gpu_add import bits, ic, pair_check  # noqa: F401  (ic: the fixture)

pytestmark = pytest.mark.gpu


def half_slope(lim, a, b):
    same = ((a > 0) & (b > 0)) | ((a < 0) & (b < 0))
    with np.errstate(all="ignore"):
        if lim == I.LIM_MINMOD:
            x = 0.5 * np.where(np.abs(a) < np.abs(b), a, b)
        elif lim == I.LIM_VANLEER:
            x = a * b / (a + b)
        else:
            x = 0.5 * np.sign(a) * np.minimum(np.minimum(2 * np.abs(a), 2 * np.abs(b)), 0.5 * np.abs(a + b))
    return np.where(same, x, 0.0)


def check(ic, lim, a, b):  # noqa: F811
    got, ref = pair_check(ic, a, b, lim)[:, 4], half_slope(lim, a, b)
    with np.errstate(all="ignore"):
        ulps = np.where((got == ref) | (np.isnan(got) & np.isnan(ref)), 0.0, np.abs(got - ref) / np.spacing(np.abs(ref)))
    q = np.argmax(np.where(np.isnan(ulps), np.inf, ulps))
    assert ulps[q] <= (1.0 if lim == I.LIM_VANLEER else 0.0), (ulps[q], a[q], b[q], got[q], ref[q])


@pytest.mark.parametrize("lim", [I.LIM_MINMOD, I.LIM_VANLEER, I.LIM_MC])
def test_ordinary_differences(ic, lim):  # noqa: F811
    rng = np.random.default_rng(lim)
    a = 10.0 ** rng.uniform(-12, 4, 300_000) * rng.choice([-1.0, 1.0], 300_000)
    b = a * 10.0 ** rng.uniform(-3, 3, len(a)) * rng.choice([-1.0, 1.0, 1.0], len(a))
    check(ic, lim, a, b)
    check(ic, lim, a, np.nextafter(a, 2 * a))
    check(ic, lim, a, a)


@pytest.mark.parametrize("lim", [I.LIM_MINMOD, I.LIM_VANLEER, I.LIM_MC])
@pytest.mark.parametrize("e", [0, 1, 2, 3, 4, 30, 150, 290, 310, 690, 995, 1200, 1330, 1530, 2020, 2044, 2045, 2046])
def test_range(ic, lim, e):  # noqa: F811
    """Differences of biased exponent e with partners a few binades away and over the whole range below."""
    rng = np.random.default_rng(e)
    a = bits(rng, np.full(6000, e))
    near = np.clip(e + rng.integers(-4, 5, 3000), 0, 2046)
    b = np.abs(bits(rng, np.concatenate([near, rng.integers(0, 2047, 3000)])))
    check(ic, lim, a, np.copysign(b, a))
    check(ic, lim, np.copysign(b, a), a)


@pytest.mark.parametrize("lim", [I.LIM_MINMOD, I.LIM_VANLEER, I.LIM_MC])
def test_infinite_and_zero(ic, lim):  # noqa: F811
    v = np.array([0.0, 5e-324, 1e-320, 1e-300, 1.0, 1e300, 2.0 ** 1022, 2.0 ** 1023, np.finfo(np.float64).max, np.inf])
    v = np.concatenate([v, -v])
    a, b = (x.ravel().copy() for x in np.meshgrid(v, v))
    check(ic, lim, a, b)
