"""Convolution operands off the boundaries that the kernels read at are refused
before anything reaches the device (so this runs without a GPU): BF16 tensors
are read in pairs, an x of the weight gradient in 16 bytes."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def lib():
    from paper_1606_00556_gb300.buildlib import build
    build()
    import paper_1606_00556_gb300 as bo
    return bo


# A context that is only looked at once the operands are accepted: its device number is none that exists.
CTX = (ctypes.c_int * 64)(*([1 << 20] * 64))
DIMS = (4, 3, 2, 1)


def _call(bo, name, *args):
    return getattr(bo.lib(), name)(ctypes.cast(CTX, ctypes.c_void_p), *DIMS, *args)


A = 1 << 20  # an aligned address


@pytest.mark.parametrize("which", range(6))
@pytest.mark.parametrize("off", [1, 2, 3])
def test_forward(lib, which, off):
    p = [A, A, A, A, A, A]
    p[which] += off
    x, w, bias, res, y, yf = p
    assert _call(lib, "bo_conv3d_forward", 32, 32, x, w, bias, res, 1, y, yf) == lib.BO_ERR_ARG
    assert _call(lib, "bo_conv3d_forward", 32, 32, A, A + 4, A + 8, A, 1, A + 12, A) == lib.BO_ERR_CUDA


@pytest.mark.parametrize("which", range(3))
@pytest.mark.parametrize("off", [1, 2, 3])
def test_backward_data(lib, which, off):
    p = [A, A, A]
    p[which] += off
    assert _call(lib, "bo_conv3d_backward_data", 32, 32, *p) == lib.BO_ERR_ARG
    assert _call(lib, "bo_conv3d_backward_data", 32, 32, A + 4, A + 8, A + 12) == lib.BO_ERR_CUDA


@pytest.mark.parametrize("off", [2, 4, 8])
def test_backward_weights(lib, off):
    assert _call(lib, "bo_conv3d_backward_weights", 32, 32, A + off, A, A, A) == lib.BO_ERR_ARG
    for which in range(1, 4):
        p = [A, A, A, A]
        p[which] += 2
        assert _call(lib, "bo_conv3d_backward_weights", 32, 32, *p) == lib.BO_ERR_ARG
    assert _call(lib, "bo_conv3d_backward_weights", 32, 32, A, A + 4, A + 8, A + 12) == lib.BO_ERR_CUDA
