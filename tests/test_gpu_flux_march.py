"""Single-precision theta / phi fluxes by marching threads against the FP64 oracle at the ends of their
chunks (4 faces where the columns are few: 11 .. 33 faces leave every remainder), one cell along phi and
radial sizes that end inside a block. One step, 2e-5 of each field's scale: the bar of the
single-precision parity tests."""
import pytest

from paper_2501_15923_gb300 import inputs as I

from .test_gpu_parity import field_errors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("limiter,flux", [(I.LIM_VANLEER, I.FLUX_TVDLF), (I.LIM_MINMOD, I.FLUX_HLL)])
@pytest.mark.parametrize("shape", [(33, 10, 1), (129, 15, 2), (31, 16, 17), (5, 17, 31), (64, 32, 18)])
def test_march_against_oracle(prec, limiter, flux, shape):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle.oracle import from_workload
    from paper_2501_15923_gb300 import build
    build.build()
    from paper_2501_15923_gb300 import icarus as ic
    w = I.dynamic_cme(3, grid=I.Grid(*shape), days=2.0)
    w.opts = I.Options(limiter=limiter, flux=flux)
    g, o = ic.from_workload(w, precision=prec), from_workload(w)
    U, t = g.get_state()
    U = I.perturbed_state(U.shape, 11, U)
    g.set_state(U, t)
    o.set_state(U, t)
    g.step(1)
    o.step()
    assert field_errors(g.get_state()[0], o.get_state()[0]).max() <= 2e-5
    g.close()
