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


def test_totals_beyond_fp32_and_nan():
    col = _column((20, 12, 8), 0x3F, lbm.LBM_STORE_F32, 1.0)
    f = lbm.lbm_get_populations(col.ctx)
    f[:1920] = 3e38            # rest populations: their FP32 sum overflows
    lbm.lbm_set_populations(col.ctx, f)
    assert abs(lbm.lbm_get_totals(col.ctx)[0] / (1920 * 3e38) - 1.0) < 1e-6
    f[100] = np.inf
    lbm.lbm_set_populations(col.ctx, f)
    assert lbm.lbm_get_totals(col.ctx)[0] == np.inf
    f[100] = np.nan
    lbm.lbm_set_populations(col.ctx, f)
    assert np.isnan(lbm.lbm_get_totals(col.ctx)).all()
    col.close()
