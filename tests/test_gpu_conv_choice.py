"""tpfnet_conv3x3_tcgen05 and tpfnet_conv3x3_wgrad_tcgen05 against the kernels that run (needs a
GB300; kernel names by torch.profiler), and the results of the layers of extents that do not
divide into blocks and whose channels do not fit beside each other in shared memory."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# extents that divide into blocks, ones that do not, few pixels; narrow and wide layers, more
# tiles than SMs and fewer
SHAPES = [(4, 64, 256, 64, 64), (4, 16, 64, 256, 256), (4, 32, 128, 384, 128), (1, 33, 32, 32, 64),
          (6, 107, 330, 32, 32), (1, 31, 40, 256, 256), (8, 30, 120, 128, 128), (4, 15, 60, 256, 256),
          (2, 60, 250, 192, 64), (4, 30, 120, 384, 128), (1, 20, 52, 768, 32), (1, 20, 52, 800, 32),
          (2, 6, 80, 64, 96), (1, 31, 33, 64, 64), (1, 33, 33, 64, 64), (1, 4, 64, 64, 64)]


def _kernels(call):
    from torch.profiler import ProfilerActivity, profile

    for _ in range(2):  # (the first profile of a process may miss its kernels)
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            call()
            torch.cuda.synchronize()
        names = [e.key for e in p.key_averages() if "k_conv3x3" in e.key]
        if names:
            break
    return names


def test_queries_tell_what_runs():
    from paper_2306_11320_gb300.unet import net_library

    lib, p = net_library(), lambda t: C.c_void_p(t.data_ptr())  # noqa: E731
    wrong = []
    for N, H, W, Cin, Cout in SHAPES:
        g = torch.Generator(device="cuda").manual_seed(Cin + W)
        rnd = lambda *s: torch.randn(s, device="cuda", generator=g).to(torch.bfloat16)  # noqa: E731
        x, wt, dz = rnd(N, H, W, Cin), rnd(9, Cout, Cin), rnd(N, H, W, Cout)
        y, dw = torch.empty_like(dz), torch.zeros((9, Cout, Cin), device="cuda")
        fwd = _kernels(lambda: lib.tpfnet_conv3x3(p(x), N, H, W, Cin, p(wt), None, Cout, 0, p(y), None))
        if not fwd:
            pytest.skip("no kernel names from the profiler here")
        wg = _kernels(lambda: lib.tpfnet_conv3x3_wgrad(p(x), p(dz), N, H, W, Cin, Cout, p(dw), None, None))
        said = lib.tpfnet_conv3x3_tcgen05(N, H, W, Cin, Cout), lib.tpfnet_conv3x3_wgrad_tcgen05(N, H, W, Cin, Cout)
        ran = any("halo" in k or "_tc<" in k for k in fwd), any("wgrad_tc" in k for k in wg)
        if (said[0] > 0, said[1] == 1) != ran:
            wrong.append(((N, H, W, Cin, Cout), said, fwd, wg))
        # a float32 sum of n terms is within n 2^-24 sum |terms|, a stored bf16 within 2^-8
        F = torch.nn.functional
        k = wt.double().view(3, 3, Cout, Cin).permute(2, 3, 0, 1).contiguous()
        xd = x.double().permute(0, 3, 1, 2).contiguous()
        ref, mag = F.conv2d(xd, k, padding=1), F.conv2d(xd.abs(), k.abs(), padding=1)
        err = (y.double().permute(0, 3, 1, 2) - ref).abs()
        assert bool((err <= 9 * Cin * 2.0 ** -24 * mag + 2.0 ** -8 * ref.abs()).all()), (N, H, W, Cin, Cout)
    assert not wrong, wrong
