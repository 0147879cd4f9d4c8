"""The 1D complex64 step loop under Eq. (DJ)."""
import numpy as np
import pytest

from gpu_util import make_pair, relerr
from oracle import oracle as O
from paper_2009_13507_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [17, 131, 256, 257, 1000, 1024])
@pytest.mark.parametrize("steps", [1, 2, 25])
def test_fixed_magnetisation_in_the_loop(nx, steps):
    """The component factors of Eq. (DJ), formed by one warp and read by all: the lines on both
    sides of the rule, the longest line; a call whose only step is its last, and calls that follow one another. The
    bound is the precision form's 1e-5."""
    prob, s = make_pair(1, nx, 1, dx=0.1, c0=20.0, c2=-0.8, so_type=0, omega=0.3, dt=1e-3, renorm=2, mag=0.2, precision="c64")
    psi = I.random_state((3, 1, nx), nx, 0.1, 10.0) * 1.3
    s.set_state(psi)
    s.step_imag(steps)
    s.step_imag(steps)
    ref = O.step(prob, psi, 2 * steps, True)
    assert relerr(s.get_state(), ref) < 1e-5
    N = s.normalize()
    assert abs(N[0] + N[1] + N[2] - 1.0) < 1e-5 and abs(N[0] - N[2] - 0.2) < 1e-5
