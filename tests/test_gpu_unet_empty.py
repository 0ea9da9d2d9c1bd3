"""Empty batches of the U-Net's element-wise calls (needs a GB300): no images, no rows and no
channels are no error and leave the output alone, in the forms with eight channels per thread
and with one."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N,H,W,Cc", [(0, 8, 16, 32), (0, 8, 16, 3), (2, 0, 16, 32), (2, 8, 0, 32), (2, 8, 16, 0)])
def test_nothing_to_do(N, H, W, Cc):
    from paper_2306_11320_gb300.unet import net_library

    lib = net_library()
    a = torch.ones(4096, dtype=torch.bfloat16, device="cuda")
    b = torch.full((4096,), 2.0, dtype=torch.bfloat16, device="cuda")
    p, q = C.c_void_p(a.data_ptr()), C.c_void_p(b.data_ptr())
    px = N * H * W
    codes = dict(pool=lib.tpfnet_pool(p, N, H, W, Cc, q, None),
                 pool_back=lib.tpfnet_pool_back(p, N, H, W, Cc, q, 0, None),
                 pool_back_add=lib.tpfnet_pool_back(p, N, H, W, Cc, q, 1, None),
                 up_into=lib.tpfnet_up_into(p, N, H, W, Cc, q, Cc + 8, 8, None),
                 up_back=lib.tpfnet_up_back(p, N, H, W, Cc + 8, 8, Cc, q, None),
                 channels=lib.tpfnet_channels(p, Cc + 8, 8, px, Cc, q, Cc, 0, 0, None),
                 relu_mask=lib.tpfnet_relu_mask(q, p, px * Cc, None))
    torch.cuda.synchronize()
    assert not any(codes.values()), codes
    assert bool((b == 2.0).all())
