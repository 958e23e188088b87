"""FP64 flux tiles against the oracle where they can go wrong: the edges of the radial tile (31 faces a
warp) and of the theta / phi tiles (15 faces), fields that are exactly zero or uniform (the zero sums
of the integer additions) and magnitudes whose products leave the estimates' range (the library
operations). One step per state; the bar is the FP64 parity bar of test_gpu_parity (1e-12 of each
field's scale)."""
import numpy as np
import pytest

from paper_2501_15923_gb300 import inputs as I
from tests.helpers import cart_grid, opts

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


def errors(a, b):
    s = np.array([np.abs(b[0]).max()] + [np.abs(b[1:4]).max()] * 3 + [np.abs(b[4]).max()] + [np.abs(b[5:8]).max()] * 3)
    return np.abs(a - b).reshape(8, -1).max(1) / np.maximum(s, 1e-300)


@pytest.mark.parametrize("limiter,flux", [(I.LIM_VANLEER, I.FLUX_TVDLF), (I.LIM_MC, I.FLUX_TVDLF), (I.LIM_VANLEER, I.FLUX_HLL)])
@pytest.mark.parametrize("grid", [(29, 13, 14), (30, 14, 15), (31, 15, 16), (62, 29, 8), (63, 30, 30), (7, 31, 31)])
@pytest.mark.parametrize("perturbed", [False, True])
def test_tile_edges(ic, grid, limiter, flux, perturbed):
    from oracle.oracle import from_workload
    w = I.dynamic_cme(5, grid=I.Grid(*grid), days=2.0)
    w.opts = opts(limiter=limiter, flux=flux)
    g, o = ic.from_workload(w), from_workload(w)
    U, t = g.get_state()                          # the initial wind: v_theta = B_theta = 0, v_r constant in r
    if perturbed:
        U = I.perturbed_state(U.shape, 3, U)
        U[2] += 1e-2 * U[1] * np.linspace(-1, 1, U[2].size).reshape(U[2].shape)
    for _ in range(2):
        g.set_state(U, t)
        o.set_state(U, t)
        g.step(1)
        o.step()
        (U, t), (Uo, to) = g.get_state(), o.get_state()
        assert errors(U, Uo).max() <= 1e-12 and abs(t - to) <= 1e-13 * to
    g.close()


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -300, 2.0 ** 160])
def test_magnitudes(ic, scale):
    """Velocities of order s and fields of order s in a periodic box (p, B^2 ~ s^2): small s takes the
    products of differences out of the estimates' range."""
    from oracle.oracle import Oracle
    n = (33, 6, 5)
    grid, op = cart_grid(*n), opts(rho_floor=0.0, p_floor=0.0, gravity=0)
    rng = np.random.default_rng(4)
    x = np.linspace(0, 2 * np.pi, n[0], endpoint=False)
    shape = (n[2], n[1], n[0])
    rho = 1 + 0.2 * np.sin(x) + 0.01 * rng.uniform(-1, 1, shape)
    v = scale * (0.3 * np.cos(x) + 0.05 * rng.uniform(-1, 1, (3,) + shape))
    b = scale * (0.2 * np.sin(2 * x) + 0.05 * rng.uniform(-1, 1, (3,) + shape))
    p = scale ** 2 * (1 + 0.1 * np.cos(x) + 0.01 * rng.uniform(-1, 1, shape))
    e = p / (5.0 / 3 - 1) + 0.5 * rho * (v ** 2).sum(0) + 0.5 * (b ** 2).sum(0)
    U = np.stack([rho, *(rho * v), e, *b])
    g = ic.Solver(grid, 5.0 / 3, 0.0, op)
    o = Oracle(grid, 5.0 / 3, 0.0, op)
    g.set_state(U, 0.0)
    o.set_state(U, 0.0)
    g.step(1)
    o.step()
    Ug, Uo = g.get_state()[0], o.get_state()[0]
    assert np.isfinite(Uo).all()
    s = np.array([1.0, scale, scale, scale, scale ** 2, scale, scale, scale])
    assert (np.abs(Ug - Uo).reshape(8, -1).max(1) / s).max() <= 1e-12
    g.close()
