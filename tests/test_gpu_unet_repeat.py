"""Training gives the same weights on every run (needs a GB300): parameter gradients are partial
sums added up in one order; and those sums against float64 and against the atomics' form."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _p(t):
    return C.c_void_p(t.data_ptr())


@pytest.mark.parametrize("N,H,W", [(1, 64, 128), (3, 128, 512), (2, 72, 192)])
def test_two_runs_are_equal(N, H, W):
    """(levels in segments, in blocks, and of few pixels)"""
    from paper_2306_11320_gb300.unet import UNet

    g = torch.Generator(device="cuda").manual_seed(N)
    x = torch.randn((N, H, W, 32), device="cuda", generator=g).to(torch.bfloat16)
    y = torch.randn((N, H, W, 5), device="cuda", generator=g)
    runs = []
    for _ in range(2):
        net = UNet(4, 5, seed=3)
        for _ in range(3):
            net.train_step(x, y)
        assert len(net.parts) == 15
        runs.append(net)
    for k in runs[0].G:
        assert torch.equal(runs[0].G[k], runs[1].G[k]) and torch.equal(runs[0].P[k], runs[1].P[k]), k


def test_gradients_accumulate():
    """Two backward passes add up, also for a head that has no partial sums (9 outputs)."""
    from paper_2306_11320_gb300.unet import UNet

    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn((1, 8, 64, 32), device="cuda", generator=g).to(torch.bfloat16)
    net = UNet(4, 9, seed=3)
    out = net.forward(x)
    assert len(net.parts) == 14
    d = torch.randn(out.shape, device="cuda", generator=g)
    net.zero_grad()
    net.backward(d)
    once = {k: v.clone() for k, v in net.G.items()}
    net.backward(d)
    for k, v in once.items():
        assert float((net.G[k] - 2 * v).norm()) <= 1e-5 * float(v.norm()), k


@pytest.mark.parametrize("n,counts,parts,pad", [(1, [1], [1], 3), (3, [5, 256, 257], [8, 1, 305], 3),
                                                (32, [33] * 32, [7] * 32, 3),
                                                # four words per thread
                                                (4, [4, 1024, 1028, 32], [1, 8, 51, 9], 4), (2, [1024, 8], [64, 65], 4)])
def test_sum_parts(n, counts, parts, pad):
    """The nearest float32 to the exact sum but for one rounding (and 2^-46 of the terms' size,
    the rounding of the carried errors)."""
    from paper_2306_11320_gb300.unet import net_library

    lib = net_library()
    g = torch.Generator(device="cuda").manual_seed(n)
    ps = [torch.randn((q, c + pad), device="cuda", generator=g) * 10.0 ** torch.randint(-3, 4, (q, 1), device="cuda", generator=g)
          for c, q in zip(counts, parts)]
    ds = [torch.randn(c + 1, device="cuda", generator=g) for c in counts]
    want = [d[:c].double() + p[:, :c].double().sum(0) for d, p, c in zip(ds, ps, counts)]
    size = [d[:c].double().abs() + p[:, :c].double().abs().sum(0) for d, p, c in zip(ds, ps, counts)]
    keep = [float(d[-1]) for d in ds]
    vp, ll, ip = C.c_void_p, C.c_longlong, C.c_int
    args = ((vp * n)(*[t.data_ptr() for t in ps]), (ll * n)(*[c + pad for c in counts]), (ip * n)(*counts),
            (ip * n)(*parts), (vp * n)(*[t.data_ptr() for t in ds]))
    assert lib.tpfnet_sum_parts(n, *args, None) == 0
    for d, w, z, c, e in zip(ds, want, size, counts, keep):
        assert bool(((d[:c].double() - w).abs() <= 2.0 ** -24 * w.abs() + (parts[0] + 400) * 2.0 ** -46 * z).all())
        assert float(d[-1]) == e  # nothing beyond a range is written
    assert lib.tpfnet_sum_parts(33, *args, None) == -1 and lib.tpfnet_sum_parts(0, *args, None) == -1


# one split and many; half boxes; both input widths; blocks that reach past the image; mma.sync
@pytest.mark.parametrize("N,H,W,Cin,Cout", [(1, 2, 64, 32, 32), (2, 8, 128, 64, 96), (1, 3, 64, 768, 768),
                                            (2, 128, 512, 32, 32), (1, 16, 8, 96, 160), (2, 31, 41, 64, 128),
                                            (2, 6, 80, 64, 96), (1, 1, 8, 32, 64)])
def test_partial_sums_of_a_layer(N, H, W, Cin, Cout):
    from paper_2306_11320_gb300.unet import net_library

    lib = net_library()
    g = torch.Generator(device="cuda").manual_seed(H + Cin)
    x = torch.randn((N, H, W, Cin), device="cuda", generator=g).relu().to(torch.bfloat16)
    dz = torch.randn((N, H, W, Cout), device="cuda", generator=g).to(torch.bfloat16)
    n = lib.tpfnet_wgrad_parts(N, H, W, Cin, Cout)
    assert n > 0
    size = 9 * Cout * Cin + Cout
    part = torch.full((n * size + 64,), float("nan"), device="cuda")
    assert lib.tpfnet_conv3x3_wgrad_part(_p(x), _p(dz), N, H, W, Cin, Cout, _p(part), None) == 0
    assert bool(part[n * size:].isnan().all())  # every partial sum is stored, and nothing else
    p = part[:n * size].view(n, size).double()
    assert not bool(p.isnan().any())
    dw, db = torch.zeros((9, Cout, Cin), device="cuda"), torch.zeros(Cout, device="cuda")
    assert lib.tpfnet_conv3x3_wgrad(_p(x), _p(dz), N, H, W, Cin, Cout, _p(dw), _p(db), None) == 0
    # the same terms, added with atomics in any order: n roundings of at most the terms' size
    tot, mag = p.sum(0), p.abs().sum(0)
    both = torch.cat((dw.reshape(-1), db)).double()
    assert bool(((both - tot).abs() <= n * 2.0 ** -24 * mag).all())
    bad = C.c_void_p(part.data_ptr() + 4)
    assert lib.tpfnet_conv3x3_wgrad_part(_p(x), _p(dz), N, H, W, Cin, Cout, bad, None) == -1


@pytest.mark.parametrize("pixels,Cc,Cout", [(1, 32, 5), (777, 64, 8), (70000, 32, 5), (300, 256, 1)])
def test_partial_sums_of_the_head(pixels, Cc, Cout):
    from paper_2306_11320_gb300.unet import net_library

    lib = net_library()
    g = torch.Generator(device="cuda").manual_seed(pixels)
    x = torch.randn((pixels, Cc), device="cuda", generator=g).to(torch.bfloat16)
    w, d = torch.randn((Cc, Cout), device="cuda", generator=g), torch.randn((pixels, Cout), device="cuda", generator=g)
    n = lib.tpfnet_head_parts(pixels, Cc, Cout)
    part = torch.full((n * (Cc + 1) * Cout + 16,), float("nan"), device="cuda")
    dx, dx2 = torch.empty_like(x), torch.empty_like(x)
    dW, db = torch.zeros_like(w), torch.zeros(Cout, device="cuda")
    assert lib.tpfnet_head_back_part(_p(x), _p(d), pixels, Cc, _p(w), Cout, _p(dx), _p(part), None) == 0
    assert lib.tpfnet_head_back_masked(_p(x), _p(d), pixels, Cc, _p(w), Cout, _p(dx2), _p(dW), _p(db), None) == 0
    assert torch.equal(dx, dx2) and bool(part[n * (Cc + 1) * Cout:].isnan().all())
    p = part[:n * (Cc + 1) * Cout].view(n, -1).double()
    both = torch.cat((dW.reshape(-1), db)).double()
    assert bool(((both - p.sum(0)).abs() <= n * 2.0 ** -24 * p.abs().sum(0)).all())
    assert lib.tpfnet_head_parts(pixels, 24, Cout) == 0 and lib.tpfnet_head_parts(pixels, Cc, 9) == 0
