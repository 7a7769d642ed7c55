"""The four-node sweep of 16-bit storage (rows of a multiple of 4 nodes) against the
two-node sweep: the same arithmetic per node, so the same bits.  An allocator whose
population buffers start 4 bytes off an 8-byte boundary takes the two-node sweep."""
import numpy as np
import pytest

from paper_1710_07073_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu


class _OffsetAllocator:
    """Device memory from torch; allocations of ``size`` bytes start 4 bytes later."""

    def __init__(self, size):
        import torch
        self.torch, self.size, self.base = torch, size, {}
        self.alloc, self.free = lbm.ALLOC_FN(self._alloc), lbm.FREE_FN(self._free)

    def _alloc(self, nbytes, _user):
        off = 4 if nbytes == self.size else 0
        p = self.torch.cuda.caching_allocator_alloc(int(nbytes) + 16) + off
        self.base[p] = off
        return p

    def _free(self, ptr, _nbytes, _user):
        self.torch.cuda.caching_allocator_delete(ptr - self.base.pop(ptr))


def _run(dims, walls, storage, scale, bubbles, offset, params, steps):
    S = int(np.prod(dims))
    col = lbm.Column(dims, 1.7, walls, storage, scale, params=params)
    alloc = _OffsetAllocator(19 * S * 2 if offset else -1)
    lbm.lbm_set_allocator(col.ctx, alloc.alloc, alloc.free)
    rho, u = workloads.random_fields(dims, seed=3, amp=1e-3, rho_amp=1e-3)
    lbm.lbm_set_fields(col.ctx, rho.reshape(-1), u.reshape(-1))
    if bubbles is not None:
        pos, vel, diam = bubbles
        lbm.lbm_set_bubbles(col.ctx, pos.reshape(-1), vel.reshape(-1), diam)
    name = lbm.lbm_sweep_kernel(col.ctx)
    lbm.lbm_step(col.ctx, steps)
    out = (lbm.lbm_get_populations(col.ctx), lbm.lbm_get_bubbles(col.ctx))
    col.close()
    assert not alloc.base
    return name, out


def _compare(dims, walls, storage, scale, bubbles=None, params=None, steps=4):
    na, (fa, ba) = _run(dims, walls, storage, scale, bubbles, False, params, steps)
    nb, (fb, bb) = _run(dims, walls, storage, scale, bubbles, True, params, steps)
    assert ",4" in na and ",4" not in nb
    assert np.array_equal(fa, fb)
    for k in ba:
        assert np.array_equal(ba[k], bb[k]), k


FORMATS = [(lbm.LBM_STORE_F16, 256.0), (lbm.LBM_STORE_BF16, 1.0)]


@pytest.mark.parametrize("storage,scale", FORMATS)
@pytest.mark.parametrize("walls", [0x3F, 0x7F, 0x30, 0x00, 0x03, 0x0C, 0x70])
@pytest.mark.parametrize("dims", [(4, 1, 1), (8, 2, 5), (36, 3, 4), (100, 9, 7), (64, 5, 33)])
def test_force_free(dims, walls, storage, scale):
    _compare(dims, walls, storage, scale)


@pytest.mark.parametrize("storage,scale", FORMATS)
@pytest.mark.parametrize("walls", [0x3F, 0x7F, 0x30, 0x00])
@pytest.mark.parametrize("dims,count", [((36, 20, 30), 3), ((64, 32, 45), 400)])
def test_with_bubbles(dims, count, walls, storage, scale):
    # count 3: the few-bubble step (overlapped); 400: the many-bubble step.
    p = lbm.lbm_default_params()
    p.g = 1e-4
    _compare(dims, walls, storage, scale, workloads.swarm(dims, count, seed=6,
                                                          bottom_fraction=0.6), p, steps=6)
