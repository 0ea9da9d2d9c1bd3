"""The many-step kernel (needs a GB300): n steps in one call leave the state that n calls
of one step leave, bit for bit.  A call of one step exchanges nothing between tiles, so the
comparison covers what the tiles send each other, the wrap of periodic axes, the boundary
rules of the tiles' edges and the return to the population buffers; the arithmetic of a
node is the same code in both, so no tolerance is needed.  Against the oracle the kernel is
covered by the parity tests, whose small lattices take it."""
import numpy as np
import pytest

from paper_2306_11320_gb300 import workloads as WL

pytestmark = pytest.mark.gpu


def _pair(nx, ny, bc_x, bc_y, storage, **opt):
    import torch

    from paper_2306_11320_gb300.tpflbm import Lattice

    p, f, _ = WL.random_state(nx, ny, seed=nx + 3 * ny, bc_x=bc_x, bc_y=bc_y, sigma_law=1)
    p.update(opt)
    out = []
    for _ in range(2):
        lat = Lattice(nx, ny, p, storage=storage, stream=torch.cuda.Stream())
        lat.init(**{k: v.astype(np.float32) for k, v in f.items()})
        out.append(lat)
    return out


def _same(a, b):
    x, y = a.get_state(), b.get_state()
    return [k for k in x if not np.array_equal(x[k], y[k])]


@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("nx,ny,bc_x,bc_y", [
    (3, 3, 0, 1),      # one tile, its own neighbour on every side
    (32, 8, 0, 0),     # exactly one tile
    (33, 9, 0, 1),     # four tiles of half the extent
    (33, 9, 1, 0),     # inlet and outflow, each in its own tile column
    (70, 4, 0, 0),     # both walls in one tile
    (31, 17, 1, 0),    # inlet and outflow in one tile column, ragged rows
    (96, 40, 0, 1),    # whole tiles, interior ones among them
    (512, 152, 0, 0),  # as many tiles as CTAs (304)
    (512, 153, 0, 0),  # one row more: one launch per step
])
def test_steps_at_once_equal_single_steps(nx, ny, bc_x, bc_y, storage):
    a, b = _pair(nx, ny, bc_x, bc_y, storage)
    for n in (2, 7, 12):  # odd and even calls end in different buffers
        a.step(n)
        for _ in range(n):
            b.step(1)
        assert a.t == b.t
        assert _same(a, b) == [], n


@pytest.mark.parametrize("opt", [dict(collision=1, trt_lambda=0.25), dict(normal_law=1)])
def test_options(opt):
    a, b = _pair(65, 33, 1, 0, 0, **opt)
    a.step(20)
    for _ in range(20):
        b.step(1)
    assert _same(a, b) == []


def test_more_steps_than_one_launch_takes():
    a, b = _pair(37, 23, 0, 0, 0)
    a.step(1025 + 1024)
    for n in (1000, 24, 1, 1024):
        b.step(n)
    assert a.t == b.t and _same(a, b) == []


def test_captured_call_replays():
    import torch

    a, b = _pair(64, 24, 1, 0, 0)
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=a.stream):
        a.step(6)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    b.step(18)
    assert _same(a, b) == []
