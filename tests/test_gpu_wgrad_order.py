"""The order of the weight gradient's sums (needs a GB300) on images whose width is a multiple
of 64: each CTA adds up its 64 x 1 segments from left to right and from top to bottom, 16
pixels at a time, and the segments go to CTAs in runs of ceil(segments / splits).  Training
depends on it (Adam's first step turns a change of a near-zero gradient into one of up to a
whole step), so it is part of the results.

dz is zero but for a few pixels, x is one.  A one that is added while the sum stands at 2^25
is lost whatever the rounding (the spacing there is 4), and so is one that 2^25 is added to; one
added after -2^25 stays.  The expected gradients are therefore whole numbers that only this order
gives."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

BIG = 2.0 ** 25


def _segment(N, H, W, k, px):
    """(image, row, column) of pixel px of segment k."""
    row, seg = divmod(k, W // 64)
    return row // H, row % H, 64 * seg + px


# N, H, W, Cin, Cout, events (segment, pixel, value) in interior pixels, expected sum
CASES = [
    # one split: 16-pixel groups of one segment, then whole segments of rows and images
    (1, 3, 64, 768, 768, [(1, 2, BIG), (1, 20, 1.0), (1, 40, -BIG), (1, 60, 1.0)], 1.0),
    (1, 3, 64, 736, 768, [(1, 2, 1.0), (1, 20, BIG), (1, 40, 1.0), (1, 60, -BIG)], 0.0),
    (2, 4, 128, 768, 704, [(2, 9, 1.0), (3, 30, BIG), (4, 9, 1.0), (10, 30, 1.0), (12, 5, -BIG), (13, 5, 1.0)], 1.0),
    # 34 splits of 31 segments: the second run's sum is one of its own
    (4, 64, 256, 64, 64, [(4, 9, BIG), (5, 9, 1.0), (30, 9, -BIG), (31, 9, 1.0), (32, 9, 1.0)], 2.0),
    # from 2^17 pixels up: 50 splits of 41
    (2, 128, 512, 32, 32, [(8, 9, BIG), (9, 9, 1.0), (40, 9, -BIG), (41, 9, 1.0)], 1.0),
]


@pytest.mark.parametrize("N,H,W,Cin,Cout,events,expected", CASES)
def test_order_of_sums(N, H, W, Cin, Cout, events, expected):
    from paper_2306_11320_gb300.unet import net_library

    lib, p = net_library(), lambda t: C.c_void_p(t.data_ptr())  # noqa: E731
    x = torch.ones((N, H, W, Cin), dtype=torch.bfloat16, device="cuda")
    dz = torch.zeros((N, H, W, Cout), dtype=torch.bfloat16, device="cuda")
    for k, px, v in events:
        n, h, w = _segment(N, H, W, k, px)
        assert 0 < h < H - 1 and 0 < w < W - 1  # every tap reads a one
        dz[n, h, w] = v
    dw = torch.zeros(9 * Cout * Cin + 1, device="cuda")
    for at in (0, 1):  # dw on the 16-byte rule and off it
        d = dw[at:at + 9 * Cout * Cin].zero_()
        assert lib.tpfnet_conv3x3_wgrad(p(x), p(dz), N, H, W, Cin, Cout, p(d), None, None) == 0
        assert bool((d == expected).all()), (float(d.min()), float(d.max()))
    assert lib.tpfnet_status() == 0
