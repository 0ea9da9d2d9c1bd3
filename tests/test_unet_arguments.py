"""Addresses and extents that no convolution kernel can take are refused before anything is
launched (CPU: the addresses are made up and never read)."""
import ctypes as C

import pytest

X, W, Y = 0x10000, 0x20000, 0x30000  # on the 16-byte rule


@pytest.mark.parametrize("x,wt,y,ldy", [(X + 2, W, Y, 32), (X + 8, W, Y, 32), (X, W + 4, Y, 32), (X, W, Y + 2, 32),
                                        (X, W, Y + 2, 64)])
def test_misaligned_tensors_are_refused(x, wt, y, ldy):
    from paper_2306_11320_gb300.unet import net_library

    lib, p = net_library(), C.c_void_p
    assert lib.tpfnet_conv3x3_into(p(x), 1, 2, 64, 32, p(wt), None, 32, 0, p(y), ldy, None) == -1
    if ldy == 32:
        assert lib.tpfnet_conv3x3(p(x), 1, 2, 64, 32, p(wt), None, 32, 0, p(y), None) == -1
        assert lib.tpfnet_conv3x3_dgrad_masked(p(x), 1, 2, 64, 32, p(wt), 32, None, p(y), None) == -1


@pytest.mark.parametrize("N,H,W", [(0, 2, 64), (1, 0, 64), (1, 2, 0), (0, 3, 7)])
def test_weight_gradient_of_no_pixels_is_refused(N, H, W):
    """(as the forward and data gradient refuse it)"""
    from paper_2306_11320_gb300.unet import net_library

    lib, p = net_library(), C.c_void_p
    wt = C.c_void_p(0x20000)
    assert lib.tpfnet_conv3x3_wgrad(p(X), p(Y), N, H, W, 32, 32, wt, None, None) == -1
