"""The names lbm_sweep_kernel reports are names of kernels in the library, as profilers show
them (no GPU needed: the host stubs carry the kernels' names)."""
import re
import subprocess

import pytest

from paper_1710_07073_gb300 import lbm


@pytest.fixture(scope="module")
def kernels(libpath):
    out = subprocess.run(["nm", "-C", libpath], capture_output=True, text=True, check=True).stdout
    return {m.replace(" ", "") for m in re.findall(r"lbm::(k_collide_stream\w*<[^()]*>)\(", out)}


@pytest.mark.parametrize("storage", [lbm.LBM_STORE_F32, lbm.LBM_STORE_F16, lbm.LBM_STORE_BF16])
@pytest.mark.parametrize("nx", [5, 6, 8])
def test_name_without_bubbles(kernels, nx, storage):
    h = lbm.lbm_create_storage(nx, 4, 4, 1.6, lbm.LBM_WALL_ALL, storage, 1.0)
    assert lbm.lbm_sweep_kernel(h) in kernels
    lbm.lbm_destroy(h)


@pytest.mark.parametrize("form", ["0,%d", "1,%d", "2,%d", "1,4,%d", "2,4,%d"])
@pytest.mark.parametrize("tab", [0, 1])
def test_names_with_bubbles(kernels, form, tab):
    # The forms include/lbm.h lists for two-way coupled bubbles.
    assert "k_collide_stream_pair<%s>" % (form % tab) in kernels
