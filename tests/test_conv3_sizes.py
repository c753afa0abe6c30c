"""Sizes beyond the products' int dimensions are refused, before anything is
launched (the pointers here are not memory)."""
import pytest


@pytest.mark.parametrize("ci,co,B,H,W", [(4, 4, 1 << 16, 1 << 8, 1 << 8),      # 2^32 pixels: 0 as an int
                                         (4, 4, 1 << 15, 1 << 8, 1 << 8),      # 2^31
                                         (4, 4, 1 << 30, 1 << 30, 1 << 30),    # past 64 bits
                                         (1 << 30, 4, 1, 8, 8)])
def test_too_many_pixels_or_channels(ci, co, B, H, W):
    from paper_2203_01462_gb300.surrogate import _nn
    L = _nn()
    p = 256
    assert L.nn_conv3_fwd(p, p, p, p, ci, co, B, H, W, 0, None, 0, None) == 1
    assert L.nn_conv3_dgrad(p, p, p, ci, co, B, H, W, 0, None) == 1
    assert L.nn_conv3_wgrad(p, p, p, ci, co, B, H, W, None, 0, None) == 1
