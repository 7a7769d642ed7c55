"""Periodic axes whose last tile is narrower than the others.

A window across such a boundary touches one tile more than its width alone tells: the
many-bubble step keeps a part of the Eq. 20 sum for every one of them (u_l, psi and the
velocities against the FP64 oracle)."""
import numpy as np
import pytest

from oracle import lattice as olat
from oracle.step import OracleSim
from paper_1710_07073_gb300 import lbm, workloads
from tests.gpu_util import params_for_oracle, rel_linf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,walls,forces,centre", [
    ((130, 16, 16), olat.ALL_WALLS & ~0x03, 0, (129.2, 6.0, 6.0)),
    ((65, 16, 20), olat.ALL_WALLS & ~0x03, 0, (64.6, 10.0, 6.0)),
    ((36, 33, 16), olat.ALL_WALLS & ~0x0C, lbm.LBM_FORCE_LIFT, (16.0, 0.9, 6.0)),
    ((66, 33, 17), 0, lbm.LBM_FORCE_LIFT, (65.2, 0.9, 16.4)),
])
def test_many_bubbles_across_a_ragged_boundary(dims, walls, forces, centre):
    # 300 bubbles of one diameter take the many-bubble step; the first 40 lie across the
    # boundary.  Bars of the parity tests for u_l and the velocities; psi follows the slip
    # u_b - u_l, a difference of the two, at ten times that.
    rng = np.random.default_rng(sum(dims))
    n, L = 300, np.array(dims, float)
    d = np.full(n, 1.5)
    pos = 0.75 + rng.random((n, 3)) * (L - 1.5)
    pos[:40] = np.mod(np.array(centre) + rng.uniform(-0.2, 0.2, (40, 3)), L)
    vel = 0.01 * rng.standard_normal((n, 3))
    rho, u = workloads.random_fields(dims, seed=4, amp=1e-2, rho_amp=1e-3)
    p = lbm.lbm_default_params()
    p.forces = forces
    col = lbm.Column(dims, 1.2, walls, params=p)
    sim = OracleSim(dims, 1.2, walls, params_for_oracle(p, 1.2))
    lbm.lbm_set_fields(col.ctx, rho.reshape(-1), u.reshape(-1))
    sim.set_fields(rho, u)
    lbm.lbm_set_bubbles(col.ctx, pos.reshape(-1), vel.reshape(-1), d)
    sim.set_bubbles(pos, vel, d)
    assert lbm.lbm_sweep_kernel(col.ctx).endswith(",1>" if dims[0] % 2 == 0 else "<0>")
    for _ in range(3):   # the first lists are made alone, the next ones by the update
        lbm.lbm_step(col.ctx, 1)
        sim.run(1)
        b = lbm.lbm_get_bubbles(col.ctx)
        assert rel_linf(b["ul"], sim.ul) < 1e-5
        assert rel_linf(b["vel"], sim.u) < 1e-5
        assert rel_linf(b["psi"], sim.psi) < 1e-4
    col.close()
