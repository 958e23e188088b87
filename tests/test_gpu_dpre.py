"""The training's pre-activation gradient with the fold of the ghost gradients inside, against the padding's
adjoint in numpy: one cell a direction (every ghost image is the same cell), edges and corners, and sizes
whose voxels take the kernel's loop more than once (1216 blocks of 64 voxels at O = 32, 128 at O = 16).
Small integers, so that every sum is exact in single precision and the folded ones (at most 27 x 8) in
BF16: no tolerance."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("O", [32, 16])
@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 5, 4), (5, 1, 4), (5, 4, 1), (2, 2, 2), (33, 7, 6), (130, 34, 36)])
def test_fold_mask_and_bias(O, shape):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2501_15923_gb300 import build
    build.build()
    from paper_2501_15923_gb300 import icarus as ic
    n1, n2, n3 = shape
    rng = np.random.default_rng(n1 + O)
    padded = (n3 + 2, n2 + 2, n1 + 2, O)
    g = rng.integers(-8, 9, padded).astype(np.float32)
    act = np.maximum(rng.integers(-4, 5, padded), 0).astype(np.float32)
    dpre, db = np.full(padded, np.nan, np.float32), np.full(O, np.nan, np.float32)
    p = lambda x: x.ctypes.data_as(C.c_void_p)  # noqa: E731
    assert ic.load().icarus_dpre_check(n1, n2, n3, O, p(g), p(act), p(dpre), p(db)) == 0
    # phi circular: the ghost planes to the opposite ends; theta and r replicate: to the edges
    f = g[1:-1].copy()
    f[-1] += g[0]
    f[0] += g[-1]
    f[:, 1] += f[:, 0]
    f[:, -2] += f[:, -1]
    f = f[:, 1:-1].copy()
    f[:, :, 1] += f[:, :, 0]
    f[:, :, -2] += f[:, :, -1]
    f = f[:, :, 1:-1]
    ref = np.zeros(padded, np.float32)
    ref[1:-1, 1:-1, 1:-1] = np.where(act[1:-1, 1:-1, 1:-1] > 0, f, 0)
    assert np.array_equal(dpre, ref)
    assert np.array_equal(db, ref.sum((0, 1, 2), dtype=np.float64))
