"""The refinement's transpose axis by axis (dense face gradients to the coarse
faces) against the oracle's: factors of 1, unequal factors, two to seven coarse
cells per axis, periodic and walled sides."""
import numpy as np
import pytest

from tests.gpu_common import Problem
from tests.test_gpu_adjoint import _gpu_grad, _oracle_grad, _weights, mr  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("walls", [0, 1])
@pytest.mark.parametrize("n,m", [((3, 3, 2), (1, 1, 1)), ((5, 4, 3), (1, 2, 5)), ((4, 7, 3), (5, 1, 2)), ((6, 3, 5), (3, 4, 1))])
def test_refinement_transpose_for_all_kinds_of_factors(mr, n, m, walls):  # noqa: F811
    p = Problem(*n, *m, gamma=1.3, walls=walls, dt=1e-3)
    wnu, wvar = _weights(3)
    _, g = _gpu_grad(mr, p, mr.MR_F64, 3, 2, wnu, wvar)
    _, gr = _oracle_grad(p, 3, wnu, wvar)
    # sums of a few hundred terms in FP64: the repository's bar for gradients
    for a, b in zip(g, gr):
        assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max()
