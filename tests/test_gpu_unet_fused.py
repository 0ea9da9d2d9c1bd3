"""The joined forms of the U-Net kernels (needs a GB300) against the separate calls they
stand for, on the same inputs: the same values in the same order of operations, so the
results are equal, element by element.  The separate calls are checked against the FP64
reference in test_gpu_unet.py."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _lib():
    from paper_2306_11320_gb300.unet import net_library

    return net_library()


def _p(t):
    return C.c_void_p(t.data_ptr())


def _rnd(*shape, seed=0):
    g = torch.Generator(device="cuda").manual_seed(seed + sum(shape))
    return torch.randn(shape, device="cuda", generator=g).to(torch.bfloat16)


def _ok(*codes):
    assert all(c == 0 for c in codes), codes


# (2, 6, 80, ...) takes the mma.sync kernel, the others the tcgen05 one
@pytest.mark.parametrize("N,H,W,Cin,Cout", [(2, 6, 80, 64, 96), (1, 2, 128, 32, 32), (2, 4, 64, 64, 64),
                                            (1, 8, 16, 96, 128)])
def test_convolution_forms(N, H, W, Cin, Cout):
    lib = _lib()
    x, wt = _rnd(N, H, W, Cin), _rnd(9, Cout, Cin, seed=1)
    b = torch.randn(Cout, device="cuda")
    # into a channel range of a wider tensor
    y = torch.empty((N, H, W, Cout), dtype=torch.bfloat16, device="cuda")
    wide = torch.zeros((N, H, W, Cout + 40), dtype=torch.bfloat16, device="cuda")
    part = wide[..., 32:32 + Cout]
    _ok(lib.tpfnet_conv3x3(_p(x), N, H, W, Cin, _p(wt), _p(b), Cout, 1, _p(y), None),
        lib.tpfnet_conv3x3_into(_p(x), N, H, W, Cin, _p(wt), _p(b), Cout, 1, _p(part), Cout + 40, None))
    assert torch.equal(part, y)
    assert not wide[..., :32].any() and not wide[..., 32 + Cout:].any()
    # flipped once, data gradient with the mask
    dz = _rnd(N, H, W, Cout, seed=2)
    f1, f2 = torch.empty_like(wt), torch.empty_like(wt)
    d1, d2, d3 = torch.empty_like(x), torch.empty_like(x), torch.empty_like(x)
    _ok(lib.tpfnet_conv3x3_dgrad(_p(dz), N, H, W, Cout, _p(wt), Cin, _p(f1), _p(d1), None))
    wp, fp = (C.c_void_p * 2)(wt.data_ptr(), wt.data_ptr()), (C.c_void_p * 2)(f1.data_ptr(), f2.data_ptr())
    ci, co = (C.c_int * 2)(Cin, Cin), (C.c_int * 2)(Cout, Cout)
    _ok(lib.tpfnet_flip_weights(2, wp, ci, co, fp, None),
        lib.tpfnet_conv3x3_dgrad_masked(_p(dz), N, H, W, Cout, _p(f2), Cin, None, _p(d3), None),
        lib.tpfnet_conv3x3_dgrad_masked(_p(dz), N, H, W, Cout, _p(f2), Cin, _p(x), _p(d2), None))
    ref = wt.flip(0).transpose(1, 2).reshape(wt.shape)
    assert torch.equal(f1, ref) and torch.equal(f2, ref)
    assert torch.equal(d3, d1)
    _ok(lib.tpfnet_relu_mask(_p(d1), _p(x), d1.numel(), None))
    assert torch.equal(d2, d1)


@pytest.mark.parametrize("N,H,W,C1,C2", [(1, 2, 2, 8, 8), (2, 6, 10, 32, 16), (1, 8, 64, 64, 32)])
def test_resampling_forms(N, H, W, C1, C2):
    lib = _lib()
    Ct = C1 + C2
    cat, g = _rnd(N, H, W, Ct), _rnd(N, H, W, Ct, seed=3)
    skip = torch.empty((N, H, W, C2), dtype=torch.bfloat16, device="cuda")
    _ok(lib.tpfnet_channels(_p(cat), Ct, C1, N * H * W, C2, _p(skip), C2, 0, 0, None))
    coarse = torch.empty((N, H // 2, W // 2, C2), dtype=torch.bfloat16, device="cuda")
    coarse2 = torch.empty_like(coarse)
    _ok(lib.tpfnet_pool(_p(skip), N, H, W, C2, _p(coarse), None),
        lib.tpfnet_pool_from(_p(cat[..., C1:]), N, H, W, C2, Ct, _p(coarse2), None))
    assert torch.equal(coarse, coarse2)
    # gradient at an encoder output: split, accumulate, mask
    d1, d2 = torch.empty_like(skip), torch.empty_like(skip)
    _ok(lib.tpfnet_channels(_p(g), Ct, C1, N * H * W, C2, _p(d1), C2, 0, 0, None),
        lib.tpfnet_pool_back(_p(coarse), N, H, W, C2, _p(d1), 1, None),
        lib.tpfnet_relu_mask(_p(d1), _p(skip), d1.numel(), None),
        lib.tpfnet_pool_back_skip(_p(coarse), N, H, W, C2, _p(g[..., C1:]), Ct, _p(cat[..., C1:]), Ct, _p(d2), None))
    assert torch.equal(d1, d2)
    up1 = torch.empty((N, H // 2, W // 2, C1), dtype=torch.bfloat16, device="cuda")
    up2, act = torch.empty_like(up1), _rnd(N, H // 2, W // 2, C1, seed=4)
    _ok(lib.tpfnet_up_back(_p(g), N, H, W, Ct, 0, C1, _p(up1), None),
        lib.tpfnet_relu_mask(_p(up1), _p(act), up1.numel(), None),
        lib.tpfnet_up_back_masked(_p(g), N, H, W, Ct, 0, C1, _p(act), _p(up2), None))
    assert torch.equal(up1, up2)


@pytest.mark.parametrize("pixels,Cin,Cout", [(1, 32, 5), (1000, 32, 8), (777, 64, 1), (300, 24, 5), (300, 32, 9)])
def test_head_forms(pixels, Cin, Cout):
    """Both forms of the head (pieces in registers; one element per thread for 24 channels
    and for 9 outputs) against float64, the masked one against the plain one.  A float32 sum
    of n terms is within n 2^-24 sum |terms| of the exact one (every bound below is that,
    element by element, plus the bf16 rounding of 2^-8 for dx)."""
    lib = _lib()
    g = torch.Generator(device="cuda").manual_seed(pixels + Cin + Cout)
    rnd = lambda *s: torch.randn(s, device="cuda", generator=g)  # noqa: E731
    x, w, b, dout = rnd(pixels, Cin).to(torch.bfloat16), rnd(Cin, Cout), rnd(Cout), rnd(pixels, Cout)
    out = torch.empty((pixels, Cout), device="cuda")
    dx, dxm = torch.empty_like(x), torch.empty_like(x)
    dW, db, dWm, dbm = (torch.zeros(s, device="cuda") for s in ((Cin, Cout), (Cout,), (Cin, Cout), (Cout,)))
    _ok(lib.tpfnet_head(_p(x), pixels, Cin, _p(w), _p(b), Cout, _p(out), None),
        lib.tpfnet_head_back(_p(x), _p(dout), pixels, Cin, _p(w), Cout, _p(dx), _p(dW), _p(db), None),
        lib.tpfnet_head_back_masked(_p(x), _p(dout), pixels, Cin, _p(w), Cout, _p(dxm), _p(dWm), _p(dbm), None))
    xd, wd, dd, u = x.double(), w.double(), dout.double(), 2.0 ** -24

    def near(got, ref, bound):
        assert ((got.double() - ref).abs() <= bound).all()

    near(out, xd @ wd + b.double(), (Cin + 1) * u * (xd.abs() @ wd.abs() + b.double().abs()))
    ref = dd @ wd.T
    near(dx, ref, 2 * Cout * u * (dd.abs() @ wd.abs().T) + 2.0 ** -8 * ref.abs())
    for W, B in ((dW, db), (dWm, dbm)):
        near(W, xd.T @ dd, pixels * u * (xd.abs().T @ dd.abs()))
        near(B, dd.sum(0), pixels * u * dd.abs().sum(0))
    assert torch.equal(dxm, torch.where(x > 0, dx, torch.zeros_like(dx)))


def test_parameters_of_the_callers_own():
    """A network whose parameters live in one tensor, and one whose gradients a caller has put
    into tensors of its own, train alike."""
    from paper_2306_11320_gb300.unet import UNet

    a, b = UNet(4, 5, seed=2), UNet(4, 5, seed=2)
    for k in b.G:
        b.G[k] = torch.zeros_like(b.G[k])
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn((1, 16, 64, 32), device="cuda", generator=g).to(torch.bfloat16)
    y = torch.randn((1, 16, 64, 5), device="cuda", generator=g)
    la, lb = a.train_step(x, y), b.train_step(x, y)
    # (the loss is an FP64 sum of one atomic per block, in any order: at most 304 roundings)
    assert abs(la - lb) <= 304 * 2.0 ** -53 * la
    for k in a.G:  # the order of the weight gradients' atomic sums is the only difference
        assert float((a.G[k] - b.G[k]).norm()) <= 1e-5 * float(a.G[k].norm()), k


# images that divide into 8 x 16 blocks: one block, two side by side, rows of blocks; channel
# counts of one chunk and several, whole and half boxes; (4, 16, 64, 256, 256) and (1, 16, 16,
# 384, 64) have too many channels for the boxes of two CTAs on an SM
@pytest.mark.parametrize("N,H,W,Cin,Cout", [(1, 16, 8, 32, 32), (1, 16, 16, 64, 64), (2, 32, 24, 96, 96),
                                            (1, 48, 40, 64, 160), (3, 16, 32, 192, 64), (1, 16, 16, 384, 64),
                                            (4, 16, 64, 256, 256), (2, 128, 256, 32, 128),
                                            # blocks that reach past the image
                                            (1, 33, 32, 32, 64), (2, 31, 17, 64, 96), (1, 107, 33, 96, 32),
                                            (3, 18, 20, 192, 128)])
def test_block_convolutions(N, H, W, Cin, Cout):
    """Forward, data and weight gradients against float64.  Bounds, element by element: a
    float32 sum of n terms is within n 2^-24 sum |terms|, a stored bf16 within 2^-8 of its
    value; weight gradients are added to what is there."""
    lib = _lib()
    x, wt, dz = _rnd(N, H, W, Cin).relu(), _rnd(9, Cout, Cin, seed=1), _rnd(N, H, W, Cout, seed=2)
    g = torch.Generator(device="cuda").manual_seed(H + W)
    b = torch.randn(Cout, device="cuda", generator=g)
    dw0, db0 = torch.randn((9, Cout, Cin), device="cuda", generator=g), torch.randn(Cout, device="cuda", generator=g)
    y, dx, wf, dw, db = torch.empty_like(dz), torch.empty_like(x), torch.empty_like(wt), dw0.clone(), db0.clone()
    _ok(lib.tpfnet_conv3x3(_p(x), N, H, W, Cin, _p(wt), _p(b), Cout, 0, _p(y), None),
        lib.tpfnet_conv3x3_dgrad(_p(dz), N, H, W, Cout, _p(wt), Cin, _p(wf), _p(dx), None),
        lib.tpfnet_conv3x3_wgrad(_p(x), _p(dz), N, H, W, Cin, Cout, _p(dw), _p(db), None))
    assert lib.tpfnet_status() == 0
    F = torch.nn.functional
    k = wt.double().view(3, 3, Cout, Cin).permute(2, 3, 0, 1).contiguous()
    xd, dd = x.double().permute(0, 3, 1, 2).contiguous(), dz.double().permute(0, 3, 1, 2).contiguous()
    u, nhwc = 2.0 ** -24, lambda t: t.permute(0, 2, 3, 1)

    def near(got, ref, mag, n, store):
        assert ((got.double() - ref).abs() <= n * u * mag + store * ref.abs()).all()

    ref, mag = F.conv2d(xd, k, b.double(), padding=1), F.conv2d(xd.abs(), k.abs(), b.double().abs(), padding=1)
    near(y, nhwc(ref), nhwc(mag), 9 * Cin + 1, 2.0 ** -8)
    ref, mag = F.conv_transpose2d(dd, k, padding=1), F.conv_transpose2d(dd.abs(), k.abs(), padding=1)
    near(dx, nhwc(ref), nhwc(mag), 9 * Cout, 2.0 ** -8)
    px = N * H * W
    pad = F.pad(xd, (1, 1, 1, 1))
    for tap in range(9):
        win = pad[:, :, tap // 3:tap // 3 + H, tap % 3:tap % 3 + W]
        ref = torch.einsum("nohw,nihw->oi", dd, win) + dw0[tap].double()
        mag = torch.einsum("nohw,nihw->oi", dd.abs(), win.abs()) + dw0[tap].double().abs()
        near(dw[tap], ref, mag, px + 1, 0.0)
    near(db, dd.sum((0, 2, 3)) + db0.double(), dd.abs().sum((0, 2, 3)) + db0.double().abs(), px + 1, 0.0)
