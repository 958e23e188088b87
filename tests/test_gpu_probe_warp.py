"""Probe sampling by one warp per probe: more probes than a block has warps, knot counts around the
32 samples of a search round, grids around them in every direction; stencil indices exact, values to
the FP64 parity bar against the oracle."""
import numpy as np
import pytest

from paper_2501_15923_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid", [(31, 12, 20), (33, 40, 70), (300, 33, 32)])
@pytest.mark.parametrize("probes,knots", [(1, 1), (5, 2), (33, 33), (70, 1100)])
def test_probes_against_oracle(grid, probes, knots):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle.oracle import from_workload
    from paper_2501_15923_gb300 import build
    build.build()
    from paper_2501_15923_gb300 import icarus as ic
    w = I.static_sheet(2, grid=I.Grid(*grid))
    rng = np.random.default_rng(probes)
    t = np.sort(rng.uniform(-5.0, 5.0, (probes, knots)), axis=1) * I.DAY
    traj = np.stack([t, rng.uniform(0.05, 2.2, t.shape) * I.AU, rng.uniform(-1.2, 1.2, t.shape), rng.uniform(-20, 20, t.shape)], 2)
    g, o = ic.from_workload(w), from_workload(w)
    for day in (0.0, 1.0, 7.0):
        U, _ = g.get_state()
        tc = day * I.DAY / g.scales()["t0"]
        g.set_state(U, tc)
        o.set_state(U, tc)
        rec, n = g.sample(traj, cap=1)
        ref = o.sample(traj)
        assert n == 1 and np.array_equal(rec[0][:, 10:], ref[:, 10:])
        scale = np.maximum(np.abs(ref[:, :10]).max(0), 1e-300)
        assert (np.abs(rec[0][:, :10] - ref[:, :10]) / scale).max() <= 1e-12
    g.close()
