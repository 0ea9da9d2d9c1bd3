"""Workspaces of tpflbm_create_in (needs a GB300): one without room for the many-step kernel's
words is taken, the lattice steps to the same state without it, bit for bit, and writes no
byte beyond; a smaller one is refused."""
import ctypes as C

import numpy as np
import pytest

from paper_2306_11320_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("nx,ny", [(64, 24), (37, 21), (3, 3), (640, 128)])
def test_workspace_without_words(nx, ny, storage):
    from paper_2306_11320_gb300.tpflbm import Lattice, load_library, make_params

    lib = load_library()
    p, f, _ = WL.random_state(nx, ny, seed=nx, bc_x=0, bc_y=0, sigma_law=1)
    if storage:
        p.update(WL.fp16_scales(p))
    f = {k: v.astype(np.float32) for k, v in f.items()}
    par = make_params(p, storage)
    full = lib.tpflbm_workspace_bytes(nx, ny, C.byref(par))
    up = lambda v: -(-v // 256) * 256  # noqa: E731
    tiles = -(-nx // 32) * -(-ny // 8)
    plane = -(-nx * ny // 64) * 64
    small = full - (up(4 * tiles) + up(288 * plane) if tiles <= 304 else 0)
    guard = 1 << 16
    ws = torch.full((small + guard,), 7, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    assert ws.data_ptr() % 256 == 0
    h = C.c_void_p()
    at = C.c_void_p(ws.data_ptr())
    assert lib.tpflbm_create_in(nx, ny, C.byref(par), at, small - 1, C.byref(h)) != 0 and not h.value
    assert lib.tpflbm_create_in(nx, ny, C.byref(par), at, small, C.byref(h)) == 0
    arrs = [f[k].ctypes.data_as(C.c_void_p) for k in ("phi", "ux", "uy", "p", "T")]
    assert lib.tpflbm_init(h, *arrs) == 0 and lib.tpflbm_step(h, 70) == 0
    got = [np.empty((n, ny, nx), dtype=np.float32) for n in (9, 9, 9, 2)]
    assert lib.tpflbm_get_state(h, *[a.ctypes.data_as(C.c_void_p) for a in got]) == 0
    lib.tpflbm_destroy(h)
    assert bool((ws[small:] == 7).all())
    lat = Lattice(nx, ny, p, storage=storage)
    lat.init(**f)
    lat.step(70)
    for a, b in zip(got, lat.get_state().values()):
        assert np.array_equal(a, b)
