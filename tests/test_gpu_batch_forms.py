"""A batch's sweep by nodes per thread: 16-bit columns whose rows are all a multiple of 4 take
four, any other batch two; and columns without two-way coupling have no tile lists."""
import numpy as np
import pytest

from paper_1710_07073_gb300 import lbm

pytestmark = pytest.mark.gpu

FOUR = [((4, 3, 5), 1.2), ((36, 10, 9), 1.7), ((64, 8, 31), 1.5)]


def _batch(cols, storage, scale, shape=None, params=None):
    b = lbm.Batch([c[0] for c in cols], [c[1] for c in cols], None, storage, scale, params=params)
    if shape:
        lbm.lbm_batch_set_launch_shape(b.h, *shape)
    pos = np.array([[0.5 * d[0], 0.5 * d[1], 0.4 * d[2]] for d, _ in cols])
    lbm.lbm_batch_set_bubbles(b.h, [1] * len(cols), pos.reshape(-1), np.full(3 * len(cols), 0.01),
                              np.full(len(cols), 1.1))
    lbm.lbm_batch_step(b.h, 5)
    out = [b.fields(c) for c in range(len(cols))], lbm.lbm_batch_get_bubbles(b.h)
    b.close()
    return out


@pytest.mark.parametrize("storage,scale", [(lbm.LBM_STORE_F16, 256.0), (lbm.LBM_STORE_BF16, 1.0)])
def test_four_nodes_equal_two(storage, scale):
    # A last column with rows of 6 keeps the whole batch at two nodes.
    two, b2 = _batch(FOUR + [((6, 8, 8), 1.4)], storage, scale)
    for shape in (None, (1, 2, 0), (2, 3, 0), (4, 1, 7)):
        four, b4 = _batch(FOUR, storage, scale, shape)
        for (r4, u4), (r2, u2) in zip(four, two):
            assert np.array_equal(r4, r2) and np.array_equal(u4, u2)
        for k in b4:
            assert np.array_equal(b4[k], b2[k][:3]), k


@pytest.mark.parametrize("storage,scale", [(lbm.LBM_STORE_F32, 1.0), (lbm.LBM_STORE_F16, 256.0)])
def test_one_way_columns_stay_at_rest(storage, scale):
    p = lbm.lbm_default_params()
    p.two_way = 0
    fields, b = _batch(FOUR, storage, scale, params=p)
    for rho, u in fields:
        assert (rho == 1.0).all() and not u.any()
    assert (b["vel"][:, 2] > 0).all()
