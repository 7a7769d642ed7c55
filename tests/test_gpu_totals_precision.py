"""The FP64 totals carry what FP64 sums carry (GPU).

Large values that cancel and small ones whose bits lie beyond two floats' 48, laid out so
that a thread of the totals' kernel meets +B, two small values and -B, one from each
quarter of the box (192 threads in 304 CTAs, a site or an x-pair each).  Every partial sum
is a multiple of 2^-53 below 1, so FP64 sums are exact and the totals have to be equal."""
import math

import numpy as np
import pytest

from paper_1710_07073_gb300 import lbm
from tests.test_gpu_readout import test_totals_against_exact_sums as _against_exact_sums

pytestmark = pytest.mark.gpu

B = 2.0 ** -6


def momentum_totals(dims, seed):
    """(lbm_get_totals[1:], the exact sums) of the layout above."""
    S = int(np.prod(dims))
    rng = np.random.default_rng(seed)
    g = (1.0 + rng.integers(0, 2 ** 23, (19, S)) * 2.0 ** -23) * 2.0 ** -30
    g[:, :S // 4] = B
    g[:, 3 * S // 4:] = -B
    c, w = lbm.lbm_velocity_set()
    col = lbm.Column(dims, 1.7, lbm.LBM_WALL_ALL)
    # w + g rounds by at most 2^-55, less than half an ulp of g in FP32: g is stored exactly.
    lbm.lbm_set_populations(col.ctx, (w[:, None] + g).reshape(-1))
    got = lbm.lbm_get_totals(col.ctx)[1:]
    col.close()
    return got, [math.fsum((c[:, a][:, None] * g).reshape(-1)) for a in range(3)]


@pytest.mark.parametrize("dims", [(114, 64, 64), (57, 64, 64)])
def test_sums_that_fp64_holds_exactly(dims):
    got, want = momentum_totals(dims, seed=dims[0])
    assert list(got) == want


@pytest.mark.parametrize("dims,storage,scale", [((57, 64, 66), lbm.LBM_STORE_F16, 256.0),
                                                ((13, 5, 7), lbm.LBM_STORE_BF16, 1.0)])
def test_odd_rows_in_16_bits(dims, storage, scale):
    _against_exact_sums(dims, 0x3F, storage, scale)


def test_odd_rows_beyond_fp32_and_nan():
    col = lbm.Column((21, 12, 8), 1.7, 0x3F)
    f = lbm.lbm_get_populations(col.ctx)
    f[:4032] = 3e38            # two directions: a site's FP32 sum overflows
    lbm.lbm_set_populations(col.ctx, f)
    assert abs(lbm.lbm_get_totals(col.ctx)[0] / (4032 * 3e38) - 1.0) < 1e-6
    for bad in (np.inf, np.nan):
        f[100] = bad
        lbm.lbm_set_populations(col.ctx, f)
        assert not np.isfinite(lbm.lbm_get_totals(col.ctx)[0])
    col.close()
