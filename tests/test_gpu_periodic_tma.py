"""The TMA-staged step on lattices that are periodic in both directions (needs a GB300), where the
CTAs that take the tiles next to the y seam sit out rounds of the others: extents that give no
such round, one, two and three, and more seam tiles than CTAs, for both storage modes.  Against
the same lattice as the only member of an ensemble on the general tile path, with the bounds of
test_gpu_ragged_tma.py: the two may round differently, a tile that no CTA took or that two did
would be far outside."""
import numpy as np
import pytest

from oracle.oracle import OracleSim
from paper_2306_11320_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

FIELDS = ("phi", "ux", "uy", "p", "T")


@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("nx,ny", [
    (4096, 24),    # one row of TMA tiles: one round
    (64, 2048),    # two
    (264, 1024),   # three; ragged columns on the seam
    (4864, 32),    # as many seam tiles as CTAs: none
    (8192, 40),    # more seam tiles than CTAs
])
def test_periodic_in_both_directions(nx, ny, storage):
    from fieldcheck import float32_spread
    from paper_2306_11320_gb300.tpflbm import Batch, Lattice

    p, f, _ = WL.random_state(nx, ny, seed=nx + ny, bc_x=0, bc_y=1, sigma_law=0)
    f["T"] = f["T"] - 0.01 * np.arange(nx)  # keep sigma(T) in range on a long lattice
    p.update(T_bot_slope=0.0, T_top_slope=0.0)
    if storage:
        p.update(WL.fp16_scales(p))
    f32 = {k: v.astype(np.float32) for k, v in f.items()}
    steps = 12
    lat = Lattice(nx, ny, p, storage=storage)
    lat.init(**f32)
    lat.step(steps)
    b = Batch([(nx, ny, p)], storage=storage)
    b.init(0, **f32)
    b.set_variant(0)
    b.step(steps)
    o = OracleSim(nx, ny, p)
    o.init(**{k: v.astype(np.float64) for k, v in f32.items()})
    o.step(steps)
    spread = float32_spread(nx, ny, p, f, steps, o.fields())
    x, y = lat.fields(), b.fields(0)
    for n in FIELDS:
        a, c = x[n].astype(np.float64), y[n].astype(np.float64)
        err = np.sqrt(((a - c) ** 2).sum() / (c ** 2).sum())
        bound = max(1e-6 if storage == 0 else 5e-3, 3.0 * spread[n])
        assert err <= bound, (n, err, bound)
