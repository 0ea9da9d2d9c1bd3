"""A lattice's set-up against the work of other streams (needs a GB300): create clears the step
counts and words of the many-step kernel and lays out tile lists on the default stream, while
the lattice runs on a stream of its own, which does not wait for that one.  A lattice created
over memory that an earlier lattice used, while the default stream is busy, has to step as one
created on an idle GPU does, bit for bit."""
import numpy as np
import pytest

from paper_2306_11320_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _state(nx, ny):
    p, f, _ = WL.random_state(nx, ny, seed=nx + ny, bc_x=0, bc_y=0, sigma_law=1)
    return p, {k: v.astype(np.float32) for k, v in f.items()}


@pytest.fixture(scope="module")
def busy():
    """Queues about a tenth of a second of matrix products on the default stream."""
    a = torch.randn((8192, 8192), device="cuda").to(torch.bfloat16)
    out = torch.empty_like(a)

    def queue():
        for _ in range(150):
            torch.matmul(a, a, out=out)

    queue()
    torch.cuda.synchronize()
    return queue


# odd rows (no tensor maps, no tile list); rows on the 16-byte rule; more tiles than the
# many-step kernel takes
@pytest.mark.parametrize("nx,ny", [(331, 117), (128, 32), (520, 200)])
@pytest.mark.parametrize("workspace", ["torch", "library"])
def test_lattice_created_behind_a_queue(nx, ny, workspace, busy):
    from paper_2306_11320_gb300.tpflbm import Lattice

    p, f = _state(nx, ny)
    states = []
    for queued in (False, True):
        first = Lattice(nx, ny, p, workspace=workspace)  # leaves its counts and words behind
        first.init(**f)
        first.step(40)
        torch.cuda.synchronize()
        first.close()
        del first
        if queued:
            busy()
        lat = Lattice(nx, ny, p, workspace=workspace, stream=torch.cuda.Stream())
        lat.init(**f)
        lat.step(33)
        states.append(lat.get_state())
        torch.cuda.synchronize()
        lat.close()
    for k in states[0]:
        assert np.array_equal(states[0][k], states[1][k]), k


def test_lattice_over_a_block_that_is_still_written(busy):
    """The workspace is torch memory: a block that a freed tensor of the current stream still has
    work queued on."""
    from paper_2306_11320_gb300.tpflbm import Lattice

    nx, ny = 331, 117
    p, f = _state(nx, ny)
    idle = Lattice(nx, ny, p)
    size = idle._ws.numel()
    idle.init(**f)
    idle.step(33)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        x = torch.empty(size, dtype=torch.uint8, device="cuda")
        where = x.data_ptr()
        busy()
        x.fill_(1)
        del x
        lat = Lattice(nx, ny, p)
        assert lat._ws.data_ptr() == where
        lat.init(**f)
        lat.step(33)
    a, b = idle.get_state(), lat.get_state()
    for k in a:
        assert np.array_equal(a[k], b[k]), k


def test_batch_created_behind_a_queue(busy):
    from paper_2306_11320_gb300.tpflbm import Batch

    sizes = [(64, 40), (96, 33), (331, 117)]
    got = []
    for queued in (False, True):
        if queued:
            busy()
        b = Batch([(nx, ny, _state(nx, ny)[0]) for nx, ny in sizes])
        for k, (nx, ny) in enumerate(sizes):
            b.init(k, **_state(nx, ny)[1])
        b.set_variant(4)
        b.step(9)
        got.append([b.fields(k) for k in range(len(sizes))])
        torch.cuda.synchronize()
    for x, y in zip(*got):
        for k in x:
            assert np.array_equal(x[k], y[k]), k
