"""Device memory of the many-bubble lists: 12 bytes of lists and 36 of interpolation sums per
(tile, bubble) entry, with lift or without."""
import numpy as np
import pytest

from paper_1710_07073_gb300 import lbm
from tests.test_gpu_pinned_outputs import _Counting

pytestmark = pytest.mark.gpu


class _Bytes(_Counting):
    total = 0

    def _alloc(self, nbytes, _user):
        self.total += nbytes
        return super()._alloc(nbytes, _user)


def _list_bytes(n, forces):
    p = lbm.lbm_default_params()
    p.forces = forces
    col = lbm.Column((64, 64, 64), 1.6, params=p)
    mem = _Bytes()
    lbm.lbm_set_allocator(col.ctx, mem.alloc, mem.free)
    lbm.lbm_set_fields(col.ctx)
    before = mem.total
    pos = np.full((n, 3), 32.0)
    lbm.lbm_set_bubbles(col.ctx, pos.reshape(-1), None, np.full(n, 6.0))
    used = mem.total - before
    col.close()
    return used


@pytest.mark.parametrize("forces", [0, lbm.LBM_FORCE_LIFT])
def test_bytes_per_entry(forces):
    # Windows of 9 + 1 cells half-width: 21 cells, at most 2 x 7 x 7 tiles; a bubble's own
    # state takes less than 512 bytes.
    per_bubble = (_list_bytes(3000, forces) - _list_bytes(1000, forces)) / 2000
    assert 98 * 48 < per_bubble < 98 * 48 + 512
