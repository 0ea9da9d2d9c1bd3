"""Layers of different shapes launched from two threads on streams of their own (needs a
GB300): every call succeeds and gives what it gives alone.  The shapes of a pair run in the
same kernel with different amounts of shared memory."""
import ctypes as C
import threading

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _p(t):
    return C.c_void_p(t.data_ptr())


class _Layer:
    def __init__(self, N, H, W, Cin, Cout):
        g = torch.Generator(device="cuda").manual_seed(Cin + Cout)
        rnd = lambda *s: torch.randn(s, device="cuda", generator=g).to(torch.bfloat16)  # noqa: E731
        self.dims = (N, H, W, Cin)
        self.co = Cout
        self.x, self.wt, self.dz = rnd(N, H, W, Cin), rnd(9, Cout, Cin), rnd(N, H, W, Cout)
        self.y = torch.empty_like(self.dz)
        self.dw = torch.zeros((9, Cout, Cin), device="cuda")

    def forward(self, lib, s):
        return lib.tpfnet_conv3x3(_p(self.x), *self.dims, _p(self.wt), None, self.co, 0, _p(self.y), s)

    def wgrad(self, lib, s):
        return lib.tpfnet_conv3x3_wgrad(_p(self.x), _p(self.dz), *self.dims, self.co, _p(self.dw), None, s)


@pytest.mark.parametrize("what,a,b", [
    ("forward", (1, 16, 16, 64, 32), (1, 16, 16, 384, 64)),   # few CTAs: a whole SM's memory
    ("forward", (2, 128, 256, 64, 64), (2, 128, 256, 128, 64)),  # two CTAs on an SM
    ("wgrad", (1, 4, 64, 64, 64), (1, 4, 64, 64, 128)),       # one dz box, two
    ("wgrad", (1, 16, 24, 32, 32), (1, 16, 24, 32, 96)),
])
def test_two_threads(what, a, b):
    from paper_2306_11320_gb300.unet import net_library

    lib = net_library()
    layers, codes = [_Layer(*a), _Layer(*b)], [set(), set()]
    alone = []
    for q in layers:
        assert getattr(q, what)(lib, None) == 0
        torch.cuda.synchronize()
        alone.append((q.y.clone(), q.dw.clone()))
        q.dw.zero_()
    torch.cuda.synchronize()
    start = threading.Barrier(2)
    calls = 3000

    def work(k):
        q, s = layers[k], torch.cuda.Stream()
        f, cs = getattr(q, what), C.c_void_p(s.cuda_stream)
        start.wait()
        for _ in range(calls):
            codes[k].add(f(lib, cs))
        s.synchronize()

    threads = [threading.Thread(target=work, args=(k,)) for k in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert codes == [{0}, {0}]
    assert lib.tpfnet_status() == 0
    for q, (y, dw) in zip(layers, alone):
        if what == "forward":
            assert torch.equal(q.y, y)
            continue
        # partial sums of at most 101 CTAs, added in any order: each sum within 101 2^-24 of
        # sum |dz| |x| of the exact one
        q.dw.zero_()
        assert q.wgrad(lib, None) == 0
        got, mag = q.dw.clone(), torch.zeros_like(q.dw)
        q.x, q.dz, q.dw = q.x.abs(), q.dz.abs(), mag
        assert q.wgrad(lib, None) == 0
        assert ((got - dw).abs() <= 2 * 101 * 2.0 ** -24 * mag).all()
