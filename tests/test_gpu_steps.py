"""Kernels at the sizes where their tiling can go wrong, against the FP64 oracle."""
import numpy as np
import pytest

from gpu_util import make_pair, relerr
from oracle import oracle as O
from paper_2009_13507_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _rand(prob, seed, env=3.0):
    cell = prob.dx * (prob.dy if prob.dim == 2 else 1.0)
    return I.random_state((3, prob.ny, prob.nx), seed, cell, env)


@pytest.mark.parametrize("imag", [True, False])
@pytest.mark.parametrize("bt", [0.02, 50.0, 5000.0])
@pytest.mark.parametrize("n", [255, 256, 257, 513])
def test_table_segments(n, bt, imag):
    """The pivot walk of the coefficient tables in segments of 256 points: it ends
    after a few points (bt = 0.02), some 130 (50) or runs past the segments' ends
    (5000). Bound: the conditioning of T, about 1 + 4 bt, times 10 roundings."""
    dx = 0.1
    prob, s = make_pair(2, n, 5, dx=dx, c0=1.0, so_type=1, gamma=0.3, dt=4.0 * dx * dx * bt)
    psi = _rand(prob, 3 + n)
    s.set_state(psi)
    s.substep("cn_x", imag)
    assert relerr(s.get_state(), O.substep(prob, psi, "cn_x", imag)) < 10 * 1.2e-16 * (1.0 + 4.0 * bt) + 1e-14
