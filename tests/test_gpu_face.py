"""The FP64 TVDLF and HLL fluxes of single faces against their definition in numpy. Finite fluxes to 1e-13 of
the face's largest term of each kind (a few tens of roundings of 2^-53, about 1e-15 each); a flux that the
definition makes NaN has to be NaN."""
import ctypes as C

import numpy as np
import pytest

from paper_2501_15923_gb300 import inputs as I

pytestmark = pytest.mark.gpu
GAMMA = 1.5


@pytest.fixture(scope="module")
def ic():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_15923_gb300 import build
    build.build()
    from paper_2501_15923_gb300 import icarus
    return icarus


def face_check(ic, wl, wr, d, flux):
    wl, wr = (np.ascontiguousarray(w, dtype=np.float64) for w in (wl, wr))
    f = np.zeros_like(wl)
    p = lambda x: x.ctypes.data_as(C.c_void_p)  # noqa: E731
    assert ic.load().icarus_face_check(len(wl), d, flux, GAMMA, p(wl), p(wr), p(f)) == 0
    return f


def side(w, d):
    """Conserved state, physical flux and fast speed of the states w [8][n]."""
    rho, v, p, b = w[0], w[1:4], w[4], w[5:8]
    bb, bv, vn, bn = (b * b).sum(0), (b * v).sum(0), v[d], b[d]
    u = np.concatenate([rho[None], rho * v, (p / (GAMMA - 1) + 0.5 * rho * (v * v).sum(0) + 0.5 * bb)[None], b])
    f = np.empty_like(u)
    f[0] = rho * vn
    f[1:4] = rho * v * vn - b * bn
    f[1 + d] += p + 0.5 * bb
    f[4] = (u[4] + p + 0.5 * bb) * vn - bn * bv
    f[5:8] = vn * b - bn * v
    f[5 + d] = 0.0
    a2, b2 = GAMMA * p / rho, bb / rho
    s = a2 + b2
    disc = s * s - 4 * a2 * (bn * bn / rho)
    return u, f, np.sqrt(0.5 * (s + np.sqrt(np.where(disc < 0, 0.0, disc))))


def reference(wl, wr, d, flux):
    """(flux [8][n], scale [n][8] of the terms that are added)."""
    with np.errstate(all="ignore"):
        (ul, fl, cl), (ur, fr, cr) = side(wl, d), side(wr, d)
        vl, vr = wl[1 + d], wr[1 + d]
        c = np.maximum(np.abs(vl) + cl, np.abs(vr) + cr)
        cmax = np.fmax(np.abs(vl) + cl, np.abs(vr) + cr)
        if flux == I.FLUX_TVDLF:
            f = 0.5 * (fl + fr) - 0.5 * c * (ur - ul)
        else:
            sl, sr = np.where(vl - cl < vr - cr, vl - cl, vr - cr), np.where(vl + cl > vr + cr, vl + cl, vr + cr)
            f = np.where(sl >= 0, fl, np.where(sr <= 0, fr, (sr * fl - sl * fr + sl * sr * (ur - ul)) / (sr - sl)))
        big = [np.fmax(np.abs(wl), np.abs(wr))[q] for q in range(8)]
        v, b = big[1] + big[2] + big[3], big[5] + big[6] + big[7]
        rho, e = big[0], big[4] / (GAMMA - 1) + 0.5 * big[0] * v ** 2 + 0.5 * b ** 2
        scale = np.stack([rho * cmax] + [rho * v * cmax + big[4] + b * b] * 3 + [e * cmax * 4] + [b * (cmax + v)] * 3)
    return f, scale


def compare(ic, wl, wr, d, flux):
    f, scale = reference(wl.T, wr.T, d, flux)
    got = face_check(ic, wl, wr, d, flux).T
    nan = np.isnan(f)
    assert np.array_equal(np.isnan(got), nan), np.argwhere(np.isnan(got) != nan)[:4]
    err = np.where(nan, 0.0, np.abs(got - f) / np.where(nan, 1.0, scale))
    assert err.max() <= 1e-13, (err.max(), np.unravel_index(err.argmax(), err.shape))


def states(rng, n, mach):
    w = np.empty((n, 8))
    w[:, 0], w[:, 4] = rng.uniform(0.2, 3.0, n), rng.uniform(0.1, 2.0, n)
    w[:, 1:4] = mach * rng.standard_normal((n, 3))
    w[:, 5:8] = 0.7 * rng.standard_normal((n, 3))
    return w


@pytest.mark.parametrize("flux", [I.FLUX_TVDLF, I.FLUX_HLL])
@pytest.mark.parametrize("d", [0, 1, 2])
@pytest.mark.parametrize("mach", [0.0, 0.5, 10.0])
def test_finite_states(ic, d, flux, mach):
    rng = np.random.default_rng(d)
    compare(ic, states(rng, 20000, mach), states(rng, 20000, mach), d, flux)


@pytest.mark.parametrize("d", [0, 1, 2])
@pytest.mark.parametrize("mach", [0.0, 0.5, 10.0])
def test_hll_nan_on_one_side(ic, d, mach):
    """A NaN in any variable of one side: the comparisons of the signal speeds are false, as in the definition,
    so the flux of a face with an undefined speed on the right is undefined."""
    rng = np.random.default_rng(10 + d)
    wl, wr = states(rng, 1600, mach), states(rng, 1600, mach)
    for q in range(16):
        (wl if q < 8 else wr)[q * 100:(q + 1) * 100, q % 8] = np.nan
    compare(ic, wl, wr, d, I.FLUX_HLL)


@pytest.mark.parametrize("flux", [I.FLUX_TVDLF, I.FLUX_HLL])
@pytest.mark.parametrize("k", [-450, -300, -260, -250, -240, 240, 251, 255, 260, 300, 450])
def test_scaled_states(ic, flux, k):
    """rho and p scaled by 4^k, B by 2^k leave the speeds as they are; the products gamma p + B^2 squared leave
    the normal range at |k| = 256."""
    rng = np.random.default_rng(20)
    for d in range(3):
        wl, wr = states(rng, 4000, 0.7), states(rng, 4000, 0.7)
        for w in (wl, wr):
            w[:, [0, 4]] *= 4.0 ** k
            w[:, 5:8] *= 2.0 ** k
        compare(ic, wl, wr, d, flux)
