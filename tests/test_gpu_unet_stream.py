"""A network on a stream of its own (needs a GB300): what train_step and mse clear, add to and
read back is ordered on that stream, whatever else the default stream is busy with.  Compared
with the same network on the default stream, over steps that leave the weights alone (lr 0),
so that every step has the same gradients."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_training_beside_a_busy_default_stream():
    from paper_2306_11320_gb300.unet import UNet

    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn((2, 16, 64, 32), device="cuda", generator=g).to(torch.bfloat16)
    y = torch.randn((2, 16, 64, 5), device="cuda", generator=g)
    m = torch.randn((8192, 8192), device="cuda").to(torch.bfloat16)
    out = torch.empty_like(m)

    def busy():  # some hundredths of a second of matrix products on the default stream
        for _ in range(60):
            torch.matmul(m, m, out=out)

    a = UNet(4, 5, seed=2)
    ref = a.train_step(x, y, lr=0.0)
    busy()
    torch.cuda.synchronize()
    busy()
    b = UNet(4, 5, seed=2, stream=torch.cuda.Stream())
    # FP64 sums of one atomic per block, in any order: at most 304 roundings
    for _ in range(3):
        busy()
        assert abs(b.train_step(x, y, lr=0.0) - ref) <= 304 * 2.0 ** -53 * ref
        busy()
        b.stream.synchronize()
        for k in a.G:  # the order of the gradients' atomic sums is the only difference
            assert float((a.G[k] - b.G[k]).norm()) <= 1e-5 * float(a.G[k].norm()), k
    busy()
    assert abs(b.mse(b.forward(x), y) - ref) <= 304 * 2.0 ** -53 * ref
