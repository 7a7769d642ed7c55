"""Many-bubble binning: tile runs of one axis against the cell-by-cell lists of the oracle,
over windows that wrap, ragged tiles and lists longer than one batch of the update."""
import numpy as np
import pytest

from oracle import binning as obin
from paper_1710_07073_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("walls", [0x3F, 0x7F, 0x30, 0x0C, 0x00])
@pytest.mark.parametrize("dims,n,dmax", [((22, 21, 23), 500, 4.0), ((33, 37, 41), 300, 6.0),
                                         ((64, 18, 50), 1100, 3.0), ((20, 40, 20), 90, 6.0)])
def test_lists_over_several_steps(dims, walls, n, dmax):
    rng = np.random.default_rng(n)
    d = rng.uniform(0.8, dmax, n)
    d = np.minimum(d, (min(dims) - 2.0) / 3.0)     # 2 n + 2 <= L on a periodic axis
    r = 0.5 * d
    pos = r[:, None] + rng.random((n, 3)) * (np.array(dims) - 2.0 * r[:, None])
    vel = 0.2 * rng.standard_normal((n, 3))
    p = lbm.lbm_default_params()
    p.two_way = 0                                   # moving bubbles, liquid at rest
    col = lbm.Column(dims, 1.2, walls, params=p)
    lbm.lbm_set_bubbles(col.ctx, pos.reshape(-1), vel.reshape(-1), d)
    for steps in (1, 1, 3):
        act = lbm.lbm_get_bubbles(col.ctx)["active"]
        lbm.lbm_step(col.ctx, steps)
        if steps > 1:
            continue
        b, bins = lbm.lbm_get_bubbles(col.ctx), lbm.lbm_get_bins(col.ctx)
        off, items = obin.tile_lists(list(b["pos"]), list(p.width_factor * d), act, dims, walls & 0x3F,
                                     bins["tile"])
        assert np.array_equal(bins["offsets"], np.array(off))
        assert np.array_equal(bins["items"], np.array(items))
    col.close()
