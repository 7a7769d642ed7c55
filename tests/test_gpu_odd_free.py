"""Odd rows without tile lists leave the sweep kernel before its force gather: the same bits
as with lists at every node that no force reaches."""
import numpy as np
import pytest

from oracle import lattice as olat
from paper_1710_07073_gb300 import lbm, workloads
from tests.gpu_util import oracle_pops_to_lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage,scale", [(lbm.LBM_STORE_F32, 1.0), (lbm.LBM_STORE_F16, 256.0),
                                           (lbm.LBM_STORE_BF16, 1.0)])
@pytest.mark.parametrize("walls", [0x3F, 0x7F, 0x30, 0x00])
@pytest.mark.parametrize("dims", [(33, 13, 40), (67, 14, 41)])
def test_same_bits_away_from_the_bubble(dims, walls, storage, scale):
    nx, ny, nz = dims
    rho, u = workloads.random_fields(dims, seed=21, amp=1e-3, rho_amp=1e-3)
    f = oracle_pops_to_lib(olat.equilibrium(rho, u))
    out = []
    for bubble in (False, True):
        p = lbm.lbm_default_params()
        p.g = 1e-4
        col = lbm.Column(dims, 1.6, walls, storage, scale, params=p)
        lbm.lbm_set_populations(col.ctx, f)
        if bubble:
            lbm.lbm_set_bubbles(col.ctx, [nx / 2, ny / 2, 20.0], [0.0, 0.0, 0.02], [2.0])
        lbm.lbm_step(col.ctx, 1)
        out.append(lbm.lbm_get_populations(col.ctx).reshape(19, nz, ny, nx))
        col.close()
    # A window of 3 cells around z = 20, one cell of streaming.
    far = np.abs(np.arange(nz) + 0.5 - 20.0) > 5.0
    assert np.array_equal(out[0][:, far], out[1][:, far])
    assert not np.array_equal(out[0][:, ~far], out[1][:, ~far])
