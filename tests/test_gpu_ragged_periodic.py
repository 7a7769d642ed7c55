"""Periodic axes whose last tile is narrower than the others.

A window across such a boundary touches one tile more than its width alone tells: the
many-bubble step keeps a part of the Eq. 20 sum for every one of them (u_l, psi and the
velocities against the FP64 oracle).  On the z axis, the overlapped few-bubble step guards
the layers of cells a bubble can reach beyond the boundary, counted in cells of the box
(the bits of plain stream order, at up to the 4 cells per step that are not flagged)."""
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


@pytest.mark.parametrize("storage,scale,nx", [
    (lbm.LBM_STORE_F32, 1.0, 32), (lbm.LBM_STORE_F32, 1.0, 33), (lbm.LBM_STORE_F16, 256.0, 32),
    (lbm.LBM_STORE_BF16, 1.0, 33)])                   # 2, 1, 4 and 1 planes per sweep block
@pytest.mark.parametrize("speeds", [[3.7], [-2.3], [3.7, -2.9]])
@pytest.mark.parametrize("nz", [25, 26, 27])
def test_guard_across_a_ragged_z_boundary(nz, speeds, storage, scale, nx):
    # A small drag keeps the speed and the force on the liquid small; the bubbles pass the
    # boundary every few steps.
    p = lbm.lbm_default_params()
    p.g, p.drag_scale = 0.0, 1e-3
    pos = np.array([[10.3, 8.1, 13.4], [22.6, 7.7, 5.2]])[:len(speeds)]
    vel = np.array([[0.0, 0.0, v] for v in speeds])
    got = []
    for plain in (True, False):
        col = lbm.Column((nx, 16, nz), 1.2, olat.ALL_WALLS & ~0x30, storage, scale, params=p)
        lbm.lbm_set_bubbles(col.ctx, pos.reshape(-1), vel.reshape(-1), np.full(len(speeds), 2.0))
        lbm.lbm_set_kernel_timing(col.ctx, plain)
        lbm.lbm_step(col.ctx, 60)
        got.append((lbm.lbm_get_populations(col.ctx), lbm.lbm_get_bubbles(col.ctx)))
        col.close()
    (f0, b0), (f1, b1) = got
    assert np.abs(b0["vel"][:, 2]).min() > 1.5 and f0.std() > 0
    assert np.array_equal(f0, f1)
    for k in b0:
        assert np.array_equal(b0[k], b1[k]), k
