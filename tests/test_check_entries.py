"""Argument checks of the entry points that expose the kernels' own arithmetic (rejected before any CUDA
call, so no GPU is needed)."""
import ctypes as C

import pytest

EINVAL = -1


@pytest.fixture(scope="module")
def lib():
    from paper_2501_15923_gb300 import build
    build.build()
    from paper_2501_15923_gb300 import icarus
    return icarus.load()


def test_pair_check(lib):
    x, y = (C.c_double * 2)(1.0, 2.0), (C.c_double * 10)()
    for args in ((0, 1, x, x, y), ((1 << 24) + 1, 1, x, x, y), (2, 3, x, x, y), (2, -1, x, x, y), (2, 1, None, x, y),
                 (2, 1, x, None, y), (2, 1, x, x, None)):
        assert lib.icarus_pair_check(*args) == EINVAL, args


def test_face_check(lib):
    w, f = (C.c_double * 16)(*([1.0] * 16)), (C.c_double * 16)()
    for args in ((0, 0, 0, 1.5, w, w, f), ((1 << 22) + 1, 0, 0, 1.5, w, w, f), (2, 3, 0, 1.5, w, w, f), (2, -1, 0, 1.5, w, w, f),
                 (2, 0, 2, 1.5, w, w, f), (2, 0, 0, 1.0, w, w, f), (2, 0, 0, 1.5, None, w, f), (2, 0, 0, 1.5, w, None, f),
                 (2, 0, 0, 1.5, w, w, None)):
        assert lib.icarus_face_check(*args) == EINVAL, args


def test_dpre_check(lib):
    a = (C.c_float * (27 * 32))()
    for args in ((0, 1, 1, 32, a, a, a, a), (1, 1, 0, 32, a, a, a, a), (1, 1, 1, 8, a, a, a, a), (4096, 4096, 4, 32, a, a, a, a),
                 (1, 1, 1, 32, None, a, a, a), (1, 1, 1, 32, a, None, a, a), (1, 1, 1, 32, a, a, None, a),
                 (1, 1, 1, 32, a, a, a, None)):
        assert lib.icarus_dpre_check(*args) == EINVAL, args


def test_captured_launches(lib):
    assert lib.icarus_captured_launches(None) == 0
