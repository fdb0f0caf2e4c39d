"""Calls a network kernel refuses say why through lbm_last_error.  The shape is
refused before any device work, so this file runs without a GPU."""
import pytest


@pytest.fixture(scope="module")
def lib():
    from paper_2209_01444_gb300 import build_ext, lbm

    build_ext.build()
    return lbm.load()


# rows that fit no run of 128 pixels, channels that are no multiple of 32
@pytest.mark.parametrize("H,W,C", [(8, 200, 32), (3, 64, 32), (8, 24, 32), (8, 128, 40)])
def test_refused_convolutions_say_why(lib, H, W, C):
    # another call's message first (NULL arguments)
    assert lib.lbm_nn_wgrad3x3(None, None, 1, 4, 64, 32, 32, None, 288, 1, None, None) != 0
    before = lib.lbm_last_error(None)
    assert lib.lbm_nn_conv3x3(256, 1, H, W, C, C, 256, 9 * C, 256, 32, None, 32, 0, 0, None) == -1  # LBM_EINVAL
    assert lib.lbm_last_error(None) == b"operation not supported" != before
