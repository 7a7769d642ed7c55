"""The adjoint on forms its per-node kernels treat apart: odd rows (a node per thread),
faces of every kind on even rows (pairs), windows at a face and across the periodic
boundary, against central differences of the FP64 oracle as in test_gpu_adjoint."""
import numpy as np
import pytest

from paper_1710_07073_gb300.adjoint import TerminalVelocityProblem
from tests.test_gpu_adjoint import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,walls,positions", [
    ((15, 14, 20), 0x3F, [[7.3, 7.1, 5.2]]),
    ((13, 16, 18), 0x30, [[0.4, 8.0, 6.0]]),                    # odd, across the x boundary
    ((16, 13, 18), 0x03, [[8.2, 0.3, 17.6]]),                   # y and z periodic, across both
    ((14, 15, 17), 0x0C, [[13.7, 3.0, 5.0], [12.9, 4.5, 7.0]]),  # two overlapping windows
    ((2, 16, 18), 0x3F, [[1.0, 8.0, 6.0]]),                     # one pair a row
])
def test_gradients_against_differences(dims, walls, positions):
    d = 2.5 if dims[0] > 4 else 1.6
    prob = TerminalVelocityProblem(dims=dims, omega=1.6, positions=np.array(positions), steps=24,
                                   checkpoint_every=7, window=6, target=8e-5, walls=walls, g=1e-5)
    _check(prob, d=d)
