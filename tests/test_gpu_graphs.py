"""Which graphs a call builds: the one-step graph only for steps that are launched one by one, the four-step
graph only once sixteen steps of the same tables and probes are reached; and that the steps are the same
whatever graphs they run through (bit-identical states and probe records)."""
import numpy as np
import pytest

from paper_2501_15923_gb300 import inputs as I

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


@pytest.mark.parametrize("probes", [False, True])
def test_graphs_built(ic, probes):
    w = I.dynamic_cme(3, grid=I.Grid(33, 10, 12), days=2.0)
    s = ic.from_workload(w)
    if probes:
        s.sample(w.traj, cap=1)
    L = s.launches_per_step
    count = lambda: ic.load().icarus_captured_launches(s.ctx) / L  # noqa: E731  in steps
    for n, built in ((0, 0), (4, 1), (4, 1), (3, 1), (4, 1), (8, 5), (4, 5), (5, 5)):
        s.step(n)
        assert count() == built, (n, count())
    maps = len(w.t_maps) - 1                          # another table size drops the graphs
    for n, built in ((20, 9), (8, 9), (3, 10)):
        s.set_boundary(w.t_maps[:maps], w.maps[:maps], w.cmes)
        s.step(n)
        assert count() == built, (n, count())
    s.set_boundary(w.t_maps, w.maps, w.cmes)
    for n, built in ((2, 11), (17, 15)):
        s.step(n)
        assert count() == built, (n, count())
    s.close()


@pytest.mark.parametrize("prec", [0, 2])
def test_same_steps(ic, prec):
    w = I.dynamic_cme(4, grid=I.Grid(40, 11, 13), days=2.0)
    got = []
    for calls in ([1] * 31, [4, 8, 5, 9, 5], [31]):
        s = ic.from_workload(w, precision=prec)
        s.sample(w.traj, cap=1)
        for n in calls:
            s.step(n)
        U, t = s.get_state()
        got.append((U, t, s.sample(None, cap=64)[0].copy()))
        s.close()
    for U, t, rec in got[1:]:
        assert np.array_equal(U, got[0][0]) and t == got[0][1] and np.array_equal(rec, got[0][2])
