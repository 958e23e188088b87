"""The FP64 flux kernels' additions on the integer pipe, compared bit for bit with IEEE addition: random
exponents, near cancellation, every exponent gap around the 53 + 10 bits that are kept, ties of the
rounding, signed zeros, subnormals, the top of the range, infinities and NaN (any NaN for a NaN). Exact,
so there is no tolerance."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ic():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_15923_gb300 import build
    build.build()
    from paper_2501_15923_gb300 import icarus
    return icarus


def pair_check(ic, a, b, limiter=1):
    """[n][5]: a + b, a - b, both again (shared alignment), half the slope of the differences a and b."""
    a, b = (np.ascontiguousarray(x, dtype=np.float64) for x in (a, b))
    y = np.zeros((len(a), 5))
    p = lambda x: x.ctypes.data_as(C.c_void_p)  # noqa: E731
    assert ic.load().icarus_pair_check(len(a), limiter, p(a), p(b), p(y)) == 0
    return y


def assert_same_bits(ic, a, b):
    y = pair_check(ic, a, b)
    with np.errstate(all="ignore"):
        ref = [a + b, a - b, a + b, a - b]
    for q, r in enumerate(ref):
        got = np.ascontiguousarray(y[:, q])
        same = (got.view(np.int64) == r.view(np.int64)) | (np.isnan(got) & np.isnan(r))
        bad = np.flatnonzero(~same)
        assert bad.size == 0, (q, bad.size, a[bad[0]], b[bad[0]], got[bad[0]], r[bad[0]])


def bits(rng, exponent):
    """Doubles of the given biased exponents with random signs and mantissas."""
    n = len(exponent)
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    s = rng.integers(0, 2, n, dtype=np.uint64) << np.uint64(63)
    return (s | exponent.astype(np.uint64) << np.uint64(52) | m).view(np.float64)


def test_any_exponents(ic):
    rng = np.random.default_rng(1)
    n = 400_000
    assert_same_bits(ic, bits(rng, rng.integers(0, 2047, n)), bits(rng, rng.integers(0, 2047, n)))


@pytest.mark.parametrize("top", [1, 30, 63, 64, 65, 100, 1023, 1964, 1965, 2046])
def test_exponent_gaps(ic, top):
    """Gaps 0 .. 70 below the larger exponent, both sides of the exponents where the FP64 pipe takes over."""
    rng = np.random.default_rng(top)
    gap = np.repeat(np.arange(71), 1000)
    a, b = bits(rng, np.full(len(gap), top)), bits(rng, np.maximum(top - gap, 0))
    swap = rng.random(len(gap)) < 0.5
    assert_same_bits(ic, np.where(swap, a, b), np.where(swap, b, a))


def test_near_cancellation_and_ties(ic):
    rng = np.random.default_rng(2)
    a = bits(rng, rng.integers(60, 1970, 200_000))
    steps = rng.integers(-3, 4, len(a))
    near = (a.view(np.int64) + steps).view(np.float64)
    assert_same_bits(ic, a, -near)                     # a few ulps left, or exactly zero
    m = np.ldexp(1.0 + rng.integers(0, 1 << 52, 100_000) * 2.0 ** -52, 0)
    for half in (2.0 ** -53, 3 * 2.0 ** -54, 2.0 ** -53 * (1 - 2.0 ** -52), 2.0 ** -53 * (1 + 2.0 ** -52)):
        assert_same_bits(ic, m, np.full_like(m, half))  # ties and their neighbours on either side
        assert_same_bits(ic, m, np.full_like(m, -half))


def test_special_values(ic):
    tiny, big = np.finfo(np.float64).tiny, np.finfo(np.float64).max
    quiet = np.array([0x7ff8000000000001, 0xfff8000000000000], dtype=np.uint64).view(np.float64)
    v = np.array([0.0, 1.0, 5e-324, 1e-310, tiny, 3 * tiny, 2.0 ** -959, big, big / 2, np.inf, np.nan, *quiet])
    v = np.concatenate([v, -v])
    a, b = (x.ravel() for x in np.meshgrid(v, v))
    assert_same_bits(ic, a.copy(), b.copy())
