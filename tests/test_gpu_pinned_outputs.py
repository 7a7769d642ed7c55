"""Field outputs in pinned memory: which ones the kernel writes in place.  An array off a
double's boundary is staged like a pageable one."""
import numpy as np
import pytest

from paper_1710_07073_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu

DIMS = (24, 20, 16)
S = 24 * 20 * 16


class _Counting:
    """Device memory from torch, counting the allocations (a staged read-out makes some)."""

    def __init__(self):
        import torch
        self.torch, self.count = torch, 0
        self.alloc, self.free = lbm.ALLOC_FN(self._alloc), lbm.FREE_FN(self._free)

    def _alloc(self, nbytes, _user):
        self.count += 1
        return self.torch.cuda.caching_allocator_alloc(int(nbytes))

    def _free(self, ptr, _nbytes, _user):
        self.torch.cuda.caching_allocator_delete(ptr)


@pytest.fixture
def column():
    col = lbm.Column(DIMS, 1.6)
    col.counting = _Counting()
    lbm.lbm_set_allocator(col.ctx, col.counting.alloc, col.counting.free)
    rho, u = workloads.random_fields(DIMS, seed=2)
    lbm.lbm_set_fields(col.ctx, rho.reshape(-1), u.reshape(-1))
    col.expected = lbm.lbm_get_fields(col.ctx)
    yield col
    col.close()


def _read(col, rho, u):
    """The staging allocations of a read-out into rho and u."""
    before = col.counting.count
    lbm.lbm_get_fields(col.ctx, out_rho=rho, out_u=u)
    assert np.array_equal(rho, col.expected[0]) and np.array_equal(u, col.expected[1])
    return col.counting.count - before


@pytest.mark.parametrize("offset,staged", [(0, 0), (8, 0), (4, 2), (1, 2)])
def test_offsets_in_a_pinned_block(column, offset, staged):
    import torch
    raw = torch.zeros(8 * (4 * S + 1), dtype=torch.uint8, pin_memory=True).numpy()
    out = raw[offset:offset + 32 * S].view(np.float64)
    assert _read(column, out[:S], out[S:]) == staged
    assert not raw[:offset].any() and not raw[offset + 32 * S:].any()


@pytest.mark.parametrize("split", [False, True])
def test_registered_ranges_that_meet(column, split):
    # Registered as a whole, or as two ranges that meet inside the array.
    import torch
    page = 65536
    size = -(-24 * S // page) * page
    raw = np.zeros(size + page, dtype=np.uint8)
    at = -raw.ctypes.data % page
    u = raw[at:at + 24 * S].view(np.float64)
    base = raw.ctypes.data + at
    parts = [(base, page), (base + page, size - page)] if split else [(base, size)]
    assert 24 * S > page
    rt = torch.cuda.cudart()
    for p, n in parts:
        assert int(rt.cudaHostRegister(p, n, 0)) == 0
    try:
        assert _read(column, np.empty(S), u) == 1      # rho alone is staged
    finally:
        for p, _ in parts:
            assert int(rt.cudaHostUnregister(p)) == 0
    u[:] = 0.0
    assert _read(column, np.empty(S), u) == 2
