"""Convolutions that no kernel takes are refused before anything is launched."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def lib():
    from paper_2001_09678_gb300 import build, mpv
    build.build()
    return mpv.load()


# 32 channels of BF16 input have the tensor-core kernel only (209 channels no longer fit);
# FP32 input and one channel have the CUDA cores' limits
@pytest.mark.parametrize("in_f32,cin,cout", [
    (0, 209, 32), (0, 300, 32), (0, 100000, 32), (1, 177, 32), (1, 100000, 1), (0, 100000, 1),
    (0, 8, 2), (1, 8, 31), (0, 0, 32)])
def test_refused(lib, in_f32, cin, cout):
    p = ctypes.c_void_p(4096)
    got = lib.mpv_cnn_conv3x3(p, in_f32, 1, cin, 8, 8, p, None, cout, 0, None, p, None)
    assert got == 1, got          # MPV_ERR_INVALID_ARG
