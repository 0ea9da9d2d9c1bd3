"""The state's FP64 sums at the edges of the read-out tiles (needs a GB300): diagnostics and
residual, which walk the lattice in tiles of 32 x 8, against float64 sums over the fields that
the lattice gives, for ragged extents, every boundary kind and both storages; and counts of
non-finite nodes on such edges.

The sums take the very float32 values that fields() gives, so those without rho c_p agree to
FP64 rounding (n 2^-53 sum |terms|); rho c_p is one float32 evaluation per node (4 2^-24 of a
term)."""
import numpy as np
import pytest

from paper_2306_11320_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

SIZES = [(3, 3, 0, 1), (33, 9, 1, 0), (31, 8, 0, 0), (96, 40, 0, 0), (65, 17, 0, 1), (333, 90, 1, 0), (640, 248, 0, 0)]


def _run(nx, ny, bc_x, bc_y, storage):
    from paper_2306_11320_gb300.tpflbm import Lattice

    p, f, _ = WL.random_state(nx, ny, seed=nx + ny, bc_x=bc_x, bc_y=bc_y, sigma_law=0)
    f["T"] = f["T"] - 0.01 * np.arange(nx)
    p.update(T_bot_slope=0.0, T_top_slope=0.0)
    if storage:
        p.update(WL.fp16_scales(p))
    lat = Lattice(nx, ny, p, storage=storage)
    lat.init(**{k: v.astype(np.float32) for k, v in f.items()})
    return lat, p


def _fields(lat):
    return {k: v.astype(np.float64) for k, v in lat.fields().items()}


@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("nx,ny,bc_x,bc_y", SIZES)
def test_diagnostics(nx, ny, bc_x, bc_y, storage):
    lat, p = _run(nx, ny, bc_x, bc_y, storage)
    lat.step(4)
    f, d = _fields(lat), lat.diagnostics()
    phi, T, ux, uy = f["phi"], f["T"], f["ux"], f["uy"]
    rcp = lambda a: 0.5 * (p["rho_l"] * p["cp_l"] + p["rho_h"] * p["cp_h"]) + 0.5 * (  # noqa: E731
        p["rho_h"] * p["cp_h"] - p["rho_l"] * p["cp_l"]) * np.clip(a, -1, 1)
    inside, x = phi < 0, np.broadcast_to(np.arange(nx), phi.shape)
    terms = dict(sum_phi=phi, sum_rcpT=rcp(phi) * T, sum_T=T, Ur_num=(phi * uy)[inside], Ur_den=phi[inside],
                 ub_num=(phi * ux)[inside], xb_num=(phi * x)[inside])
    for k, v in terms.items():
        each = 4 * 2.0 ** -24 if k == "sum_rcpT" else 0.0
        bound = (2 * nx * ny * 2.0 ** -53 + each) * np.abs(v).sum()
        assert abs(d[k] - v.sum()) <= bound, (k, d[k], v.sum(), bound)
    assert d["nonfinite"] == 0


@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("nx,ny,bc_x,bc_y", SIZES)
def test_residual(nx, ny, bc_x, bc_y, storage):
    lat, _ = _run(nx, ny, bc_x, bc_y, storage)
    dT = 0.7
    assert lat.residual(dT) == (np.inf, np.inf, 0)
    a = _fields(lat)
    for steps in (3, 5):
        lat.step(steps)
        b = _fields(lat)
        ru, rT, k = lat.residual(dT)
        du = sum(((b[n] - a[n]) ** 2).sum() for n in ("ux", "uy"))
        uu = sum((b[n] ** 2).sum() for n in ("ux", "uy"))
        assert k == steps
        assert ru == pytest.approx(np.sqrt(du) / (k * np.sqrt(uu)), rel=1e-9)
        assert rT == pytest.approx(np.sqrt(((b["T"] - a["T"]) ** 2).sum()) / (k * dT * np.sqrt(nx * ny)), rel=1e-9)
        a = b


@pytest.mark.parametrize("x,y", [(0, 0), (31, 7), (32, 8), (64, 16)])
def test_nonfinite_nodes_are_counted(x, y):
    """One population of a node that is not a number: the node's phi, and with it the
    stencils of the eight nodes around it (fewer at a wall; the x axis is periodic)."""
    nx, ny = 65, 17
    lat, _ = _run(nx, ny, 0, 0, 0)
    st = lat.get_state()
    st["f"][0, y, x] = np.nan
    lat.set_state(st)
    rows = len({min(max(y + j, 0), ny - 1) for j in (-1, 0, 1)})
    d = lat.diagnostics()
    assert d["rc"] == -4 and d["nonfinite"] == 3 * rows
