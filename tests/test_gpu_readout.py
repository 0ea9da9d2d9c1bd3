"""Reading out a state (needs a GB300): the union-find labelling on regions that its parts
have to join (spirals across the 32-node runs, combs, the periodic seams, whole rows), and
fields written straight into device memory against the same fields through host memory."""
import numpy as np
import pytest

from oracle.bubbles_ref import bubbles as ref_bubbles
from paper_2306_11320_gb300 import workloads as WL

pytestmark = pytest.mark.gpu


def _mask(kind, nx, ny):
    m = np.zeros((ny, nx), dtype=bool)
    if kind == "spiral":  # one region, one node wide, as long as the lattice allows
        x0, x1, y0, y1 = 0, nx - 1, 0, ny - 1
        m[0, :] = True
        while x1 - x0 > 3 and y1 - y0 > 3:
            m[y0:y1 + 1, x1] = True
            m[y1, x0:x1 + 1] = True
            m[y0 + 2:y1 + 1, x0] = True
            m[y0 + 2, x0:x1 - 1] = True
            x0, x1, y0, y1 = x0 + 2, x1 - 2, y0 + 2, y1 - 2
    elif kind == "comb":  # teeth joined by the last row only: trees that meet late
        m[:, ::2] = True
        m[-1, :] = True
    elif kind == "rows":  # whole rows, apart from each other
        m[1::8, :] = True
    elif kind == "edges":  # the lattice's rim: one region, or several, by the seams
        m[0, 3:-3] = m[-1, 3:-3] = True
        m[3:-3, 0] = m[3:-3, -1] = True
    return m


@pytest.mark.parametrize("bc_x,bc_y", [(0, 1), (0, 0), (1, 0)])
@pytest.mark.parametrize("kind", ["spiral", "comb", "rows", "edges"])
@pytest.mark.parametrize("nx,ny", [(31, 17), (32, 40), (65, 33)])
def test_regions(nx, ny, kind, bc_x, bc_y):
    """phi = -1 inside and 1 outside: node counts and sums are whole numbers (equal), the
    centroids FP64 sums of whole numbers over their count."""
    from paper_2306_11320_gb300.tpflbm import Lattice

    phi = np.where(_mask(kind, nx, ny), -1.0, 1.0).astype(np.float32)
    z = np.zeros_like(phi)
    lat = Lattice(nx, ny, WL.base_params(bc_x=bc_x, bc_y=bc_y))
    lat.init(phi=phi, ux=z, uy=z, p=z, T=z)
    phi = lat.fields()["phi"]  # the sum of the populations: -1 within float32 rounding
    ref = ref_bubbles(phi, z, z, periodic_x=bc_x == 0, periodic_y=bc_y == 1)
    got = lat.bubbles()
    assert len(got) == len(ref)
    key = lambda b: (b["nodes"], round(b["x_b"], 3), round(b["y_b"], 3))  # noqa: E731
    for a, b in zip(sorted(got, key=key), sorted(ref, key=key)):
        assert a["nodes"] == b["nodes"]
        assert a["sum_phi"] == pytest.approx(b["sum_phi"], rel=1e-12)
        for k, n in (("x_b", nx), ("y_b", ny)):
            d = abs(a[k] - b[k])
            assert min(d, n - d) < 1e-9, (k, a, b)


@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("nx,ny,bc_x,bc_y", [(3, 3, 0, 1), (33, 9, 1, 0), (96, 40, 0, 0), (333, 90, 0, 1)])
def test_fields_into_device_memory(nx, ny, bc_x, bc_y, storage):
    from paper_2306_11320_gb300.tpflbm import Lattice

    p, f, _ = WL.random_state(nx, ny, seed=nx, bc_x=bc_x, bc_y=bc_y)
    lat = Lattice(nx, ny, p, storage=storage)
    lat.init(**{k: v.astype(np.float32) for k, v in f.items()})
    lat.step(3)
    host, dev = lat.fields(), lat.fields(device=True)
    for k in host:
        assert np.array_equal(host[k], dev[k].cpu().numpy()), k
    # some fields only, host and device mixed
    import torch

    T, ux = torch.zeros((ny, nx), device="cuda"), np.zeros((ny, nx), dtype=np.float32)
    lat._check(lat.lib.tpflbm_get_fields(lat.h, None, ux.ctypes.data, None, None, T.data_ptr()))
    assert np.array_equal(ux, host["ux"]) and np.array_equal(T.cpu().numpy(), host["T"])
