"""Lattices stepped side by side on streams of their own (needs a GB300), from one thread and
from several: each ends in the state that it reaches alone, bit for bit, whichever kernel its
calls take meanwhile (lattices of more than half as many tiles as CTAs run at once step with
one launch per step while another's grid holds the GPU)."""
import threading

import numpy as np
import pytest

from paper_2306_11320_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _make(nx, ny, storage, seed, stream):
    from paper_2306_11320_gb300.tpflbm import Lattice

    p, f, _ = WL.random_state(nx, ny, seed=seed, bc_x=seed % 2, bc_y=0, sigma_law=1)
    if storage:
        p.update(WL.fp16_scales(p))
    lat = Lattice(nx, ny, p, storage=storage, stream=stream)
    lat.init(**{k: v.astype(np.float32) for k, v in f.items()})
    return lat


CALLS = (1030, 3, 64, 1, 200)  # odd and even, several launches, short ones

# 165 and 256 tiles (of 304 CTAs), and 16; the last one has more tiles than the kernel takes
SETS = [[(331, 117), (331, 117), (331, 117), (331, 117)], [(512, 128), (128, 32), (331, 117), (640, 128)]]


@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("sizes", SETS)
@pytest.mark.parametrize("threads", [False, True])
def test_states_equal_those_alone(sizes, storage, threads):
    alone = []
    for k, (nx, ny) in enumerate(sizes):
        lat = _make(nx, ny, storage, k, torch.cuda.Stream())
        for n in CALLS:
            lat.step(n)
        alone.append((lat.t, lat.get_state()))
    lats = [_make(nx, ny, storage, k, torch.cuda.Stream()) for k, (nx, ny) in enumerate(sizes)]
    if threads:
        def work(lat):
            for n in CALLS:
                lat.step(n)

        pool = [threading.Thread(target=work, args=(lat,)) for lat in lats]
        for t in pool:
            t.start()
        for t in pool:
            t.join()
    else:
        for n in CALLS:
            for lat in lats:
                lat.step(n)
    for lat, (t, ref) in zip(lats, alone):
        assert lat.t == t
        got = lat.get_state()
        for k in ref:
            assert np.array_equal(got[k], ref[k]), k


def test_capture_beside_a_running_grid():
    """A call captured while another lattice's grid is in flight, and a call of that lattice
    while this one captures, leave the capture whole."""
    a, b = (_make(331, 117, 0, 4, torch.cuda.Stream()) for _ in range(2))
    c = _make(331, 117, 0, 4, torch.cuda.Stream())
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    a.step(1024)
    with torch.cuda.graph(g, stream=b.stream):
        b.step(6)
        a.step(512)
        c.step(16)
    for _ in range(256):
        g.replay()
    c.step(1520)
    torch.cuda.synchronize()
    x, y, z = a.get_state(), b.get_state(), c.get_state()
    for k in x:
        assert np.array_equal(x[k], y[k]) and np.array_equal(x[k], z[k]), k
