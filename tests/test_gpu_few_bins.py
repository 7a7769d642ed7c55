"""Few-bubble binning: the lists against the oracle's cell-by-cell ones at the bubble counts
where the lanes per bubble change (a warp down to two lanes of the 256 threads)."""
import numpy as np
import pytest

from oracle import binning as obin
from paper_1710_07073_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("walls", [0x3F, 0x0C, 0x00])
@pytest.mark.parametrize("n", [1, 2, 8, 9, 16, 17, 32, 33, 64, 65, 80])
def test_lists_by_lanes_per_bubble(n, walls):
    dims = (66, 33, 47)
    rng = np.random.default_rng(n)
    d = np.full(n, 1.4)
    pos = 0.7 + rng.random((n, 3)) * (np.array(dims) - 1.4)
    p = lbm.lbm_default_params()
    p.two_way = 0                                   # moving bubbles, liquid at rest
    col = lbm.Column(dims, 1.2, walls, params=p)
    lbm.lbm_set_bubbles(col.ctx, pos.reshape(-1), 0.2 * rng.standard_normal(3 * n), d)
    for _ in range(3):
        act = lbm.lbm_get_bubbles(col.ctx)["active"]
        lbm.lbm_step(col.ctx, 1)
        b, bins = lbm.lbm_get_bubbles(col.ctx), lbm.lbm_get_bins(col.ctx)
        off, items = obin.tile_lists(list(b["pos"]), list(p.width_factor * d), act, dims,
                                     walls & 0x3F, bins["tile"])
        assert np.array_equal(bins["offsets"], np.array(off))
        assert np.array_equal(bins["items"], np.array(items))
    col.close()
