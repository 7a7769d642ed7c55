"""State read-outs of the library against sums in exact arithmetic (GPU).

The FP64 totals are compensated FP32 sums per thread: against the exact sum of the
stored values they may be off by 2^-44 of the sum of magnitudes, plus the rounding of the
populations read back (half an ulp of at most 1/3 each).
"""
import math

import numpy as np
import pytest

from paper_1710_07073_gb300 import lbm

pytestmark = pytest.mark.gpu


def _column(dims, walls, storage, scale, seed=5, amp=1e-2):
    col = lbm.Column(dims, 1.7, walls, storage=storage, scale=scale)
    rng = np.random.default_rng(seed)
    S = int(np.prod(dims))
    _, w = lbm.lbm_velocity_set()
    f = (w[:, None] * (1.0 + amp * rng.standard_normal((19, S)))).reshape(-1)
    lbm.lbm_set_populations(col.ctx, f)
    return col


@pytest.mark.parametrize("dims,walls,storage,scale", [
    ((1, 1, 1), 0x00, lbm.LBM_STORE_F32, 1.0),
    ((13, 5, 7), 0x3F, lbm.LBM_STORE_F32, 1.0),
    ((32, 16, 8), 0x7F, lbm.LBM_STORE_F16, 256.0),
    ((66, 67, 40), 0x30, lbm.LBM_STORE_BF16, 1.0),
    ((128, 96, 64), 0x3F, lbm.LBM_STORE_F32, 1.0),
])
def test_totals_against_exact_sums(dims, walls, storage, scale):
    col = _column(dims, walls, storage, scale)
    S = int(np.prod(dims))
    got = lbm.lbm_get_totals(col.ctx)
    c, w = lbm.lbm_velocity_set()
    g = lbm.lbm_get_populations(col.ctx).reshape(19, S) - w[:, None]
    mag = float(np.abs(g).sum())
    tol = 2.0 ** -44 * mag + 19 * S * 2.0 ** -54 + 2.0 ** -52 * S
    want = [S + math.fsum(g.reshape(-1))]
    want += [math.fsum((c[:, a][:, None] * g).reshape(-1)) for a in range(3)]
    assert np.abs(got - np.array(want)).max() <= tol
    col.close()


@pytest.mark.parametrize("dims", [(2, 1, 1), (2, 3, 1), (64, 1, 5), (514, 3, 33), (515, 3, 33)])
@pytest.mark.parametrize("walls", [0x00, 0x3F, 0x7F])
def test_totals_by_pairs_on_thin_and_long_rows(dims, walls):
    # Rows of one pair, single rows and planes, and passes that end inside a row.
    test_totals_against_exact_sums(dims, walls, lbm.LBM_STORE_F32, 1.0)


def test_totals_beyond_fp32_and_nan():
    col = _column((20, 12, 8), 0x3F, lbm.LBM_STORE_F32, 1.0)
    f = lbm.lbm_get_populations(col.ctx)
    f[:3840] = 3e38            # two directions: a site's FP32 sum overflows
    lbm.lbm_set_populations(col.ctx, f)
    assert abs(lbm.lbm_get_totals(col.ctx)[0] / (3840 * 3e38) - 1.0) < 1e-6
    f[100] = np.inf
    lbm.lbm_set_populations(col.ctx, f)
    assert lbm.lbm_get_totals(col.ctx)[0] == np.inf
    f[100] = np.nan
    lbm.lbm_set_populations(col.ctx, f)
    assert np.isnan(lbm.lbm_get_totals(col.ctx)).all()
    col.close()


@pytest.mark.parametrize("dims,storage,scale", [((1, 1, 1), 0, 1.0), ((13, 5, 7), 1, 256.0),
                                                ((64, 33, 20), 0, 1.0)])
def test_fields_written_in_place_equal_staged_ones(dims, storage, scale):
    import torch
    col = _column(dims, 0x3F, storage, scale)
    S = int(np.prod(dims))
    rho, u = lbm.lbm_get_fields(col.ctx)                    # pageable: staged and copied
    pin = torch.full((4 * S + 2,), -7.0, dtype=torch.float64, pin_memory=True).numpy()
    # At an offset inside a pinned block, and one array of each kind.
    lbm.lbm_get_fields(col.ctx, out_rho=pin[1:S + 1], out_u=pin[S + 1:4 * S + 1])
    assert np.array_equal(pin[1:S + 1], rho) and np.array_equal(pin[S + 1:4 * S + 1], u)
    assert pin[0] == -7.0 and pin[-1] == -7.0
    pin[:] = -7.0
    r2, _ = lbm.lbm_get_fields(col.ctx, out_u=pin[1:3 * S + 1])
    assert np.array_equal(r2, rho) and np.array_equal(pin[1:3 * S + 1], u)
    b = lbm.Batch([(12, 8, 6)], [1.5])
    br, bu = lbm.lbm_batch_get_fields(b.h, 0, 576)
    pin = torch.empty(4 * 576, dtype=torch.float64, pin_memory=True).numpy()
    lbm.lbm_batch_get_fields(b.h, 0, 576, out_rho=pin[:576], out_u=pin[576:])
    assert np.array_equal(pin[:576], br) and np.array_equal(pin[576:], bu)
    b.close()
    col.close()


@pytest.mark.parametrize("n", [1, 1024, 1025])
def test_bubble_state_by_page_and_by_copies(n):
    rng = np.random.default_rng(n)
    col = lbm.Column((64, 64, 64), 1.6)
    pos = 4.0 + 56.0 * rng.random((n, 3))
    vel = rng.standard_normal((n, 3)).astype(np.float32).astype(np.float64)
    lbm.lbm_set_bubbles(col.ctx, pos, vel, np.full(n, 2.0))
    got = lbm.lbm_get_bubbles(col.ctx)
    assert np.abs(got["pos"] - pos).max() <= 64.0 * 2.0 ** -47      # two floats
    assert np.array_equal(got["vel"], vel) and got["active"].all() and len(got["active"]) == n
    assert not got["ul"].any() and not got["psi"].any()
    few = lbm.lbm_get_bubbles(col.ctx, cap=(n + 1) // 2)
    assert np.array_equal(few["pos"], got["pos"][:(n + 1) // 2])
    col.close()
