"""The network's inputs, targets and outputs below the normal single-precision range: values and scales that
are single-precision subnormals give the same normalised numbers as ordinary ones (all values are powers
of two times small integers, so the comparisons are exact)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
N = (24, 6, 5)


@pytest.fixture(scope="module")
def ic():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_15923_gb300 import build
    build.build()
    from paper_2501_15923_gb300 import icarus
    return icarus


def network(ic, in_scale, out_scale, weights=None):
    net = ic.Closure(*N, seed=3)
    if weights is not None:
        net.set_weights(weights)
    net.set_norm(np.zeros((8, N[0])), np.full((8, N[0]), in_scale), np.full((8, N[0]), out_scale))
    return net


def integers(seed):
    return np.random.default_rng(seed).integers(-15, 16, (8, N[2], N[1], N[0])).astype(np.float64)


def device(a):
    import torch
    return torch.from_numpy(a).cuda()


def test_subnormal_scales(ic):
    import torch
    U, dU = integers(1), integers(2)
    got = []
    for k in (0, -140):                               # scales 2^-136: subnormal; values down to 2^-140
        net = network(ic, 2.0 ** (k + 4), 2.0 ** (k + 4))
        u, t = device(U * 2.0 ** k), device(dU * 2.0 ** k)
        out = torch.empty_like(u)
        net.predict(u.data_ptr(), out.data_ptr())
        torch.cuda.synchronize()
        got.append((out.cpu().numpy() * 2.0 ** -k, net.train_step(u.data_ptr(), t.data_ptr(), 1e-3)))
        net.close()
    assert np.isfinite(got[1][0]).all() and np.array_equal(got[0][0], got[1][0])
    assert got[0][1] == pytest.approx(got[1][1], rel=1e-14)     # the loss: blocks add in any order


def test_subnormal_output_and_loss(ic):
    import torch
    weights = [(np.zeros((o, 27, c), np.float32), np.zeros(o, np.float32)) for c, o in ic.LAYER_SHAPES]
    weights[3][1][:8] = 2.0 ** -130                   # the output is the last bias
    net = network(ic, 1.0, 2.0 ** 130, weights)
    u = device(integers(1))
    out = torch.empty_like(u)
    net.predict(u.data_ptr(), out.data_ptr())
    torch.cuda.synchronize()
    assert (out.cpu().numpy() == 1.0).all()
    net.close()
    weights[3][1][:8] = 0.0
    net = network(ic, 1.0, 1.0, weights)
    t = device(np.full(u.shape, 2.0 ** -70))          # (y - t)^2 = 2^-140
    assert net.train_step(u.data_ptr(), t.data_ptr(), 0.0) == pytest.approx(2.0 ** -140, rel=1e-6)
    net.close()
