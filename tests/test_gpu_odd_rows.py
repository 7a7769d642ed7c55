"""Odd rows: the overlapped update and sweep give the bits of plain stream order, and one
step over small and ragged boxes matches the FP64 oracle."""
import numpy as np
import pytest

from oracle import lattice as olat
from paper_1710_07073_gb300 import lbm, workloads
from tests.gpu_util import lib_pops_to_oracle, oracle_pops_to_lib

pytestmark = pytest.mark.gpu


def _run(dims, walls, storage, scale, plain):
    pos = np.array([[0.3 * dims[0], 0.5 * dims[1], 0.3 * dims[2]],
                    [0.6 * dims[0], 0.4 * dims[1], 0.8 * dims[2]]])
    vel = np.array([[0.0, 0.0, 0.05], [0.01, 0.0, 0.04]])
    p = lbm.lbm_default_params()
    p.g = 1e-2
    col = lbm.Column(dims, 1.6, walls, storage, scale, params=p)
    lbm.lbm_set_bubbles(col.ctx, pos.reshape(-1), vel.reshape(-1), np.array([2.0, 1.6]))
    lbm.lbm_set_kernel_timing(col.ctx, plain)
    for _ in range(3):
        lbm.lbm_step(col.ctx, 40)
    out = lbm.lbm_get_populations(col.ctx), lbm.lbm_get_bubbles(col.ctx)
    col.close()
    return out


@pytest.mark.parametrize("storage,scale", [(lbm.LBM_STORE_F32, 1.0), (lbm.LBM_STORE_F16, 256.0),
                                           (lbm.LBM_STORE_BF16, 1.0)])
@pytest.mark.parametrize("dims,walls", [((33, 16, 41), 0x3F), ((21, 17, 24), 0x0F),
                                        ((65, 18, 39), 0x70), ((13, 13, 40), 0x7F)])
def test_overlapped_steps_match_plain_order(dims, walls, storage, scale):
    (f0, b0), (f1, b1) = (_run(dims, walls, storage, scale, plain) for plain in (True, False))
    assert np.array_equal(f0, f1)
    for k in b0:
        assert np.array_equal(b0[k], b1[k]), k


@pytest.mark.parametrize("walls", [0x3F, 0x7F, 0x30, 0x00, 0x0C])
@pytest.mark.parametrize("dims", [(1, 1, 1), (3, 5, 1), (37, 4, 2), (31, 9, 11), (67, 6, 8)])
def test_one_step_matches_oracle(dims, walls):
    rho, u = workloads.random_fields(dims, seed=8, amp=1e-3, rho_amp=1e-3)
    f = olat.equilibrium(rho, u)
    col = lbm.Column(dims, 1.7, walls)
    lbm.lbm_set_populations(col.ctx, oracle_pops_to_lib(f))
    lbm.lbm_step(col.ctx, 1)
    got = lib_pops_to_oracle(lbm.lbm_get_populations(col.ctx), dims)
    # FP32 on values shifted by w rho0 (the parity tests' bound).
    assert np.abs(got - olat.lb_step(f, 1.7, walls)).max() < 2e-8
    col.close()
