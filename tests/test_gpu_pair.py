"""The pair step where its increments end: non-finite states, rough states and large increments."""
import numpy as np
import pytest

from gpu_util import make_pair
from paper_2009_13507_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _rand(prob, seed, env=3.0):
    return I.random_state((3, prob.ny, prob.nx), seed, prob.dx * prob.dy, env)


@pytest.mark.parametrize("what", ["one", "two", "inf"])
@pytest.mark.parametrize("nx,ny", [(96, 100), (200, 120)])
def test_a_non_finite_norm_suspends_the_renormalisation(nx, ny, what):
    """A NaN or infinity in the state makes the step's norm non-finite, whatever the number of such points
    in a tile, and the scale stays 1: rows that it cannot have reached (at most 12 points a
    step, taps and stencil) keep the values of the finite state's steps without
    renormalisation. No reduction but the step's own runs before they are read."""
    kw = dict(dx=0.1, c0=10.0, c2=0.5, so_type=1, gamma=0.3, omega=0.2, dt=1e-3)
    prob, s = make_pair(2, nx, ny, renorm=1, **kw)
    _, f = make_pair(2, nx, ny, renorm=0, **kw)
    psi = _rand(prob, 3, env=20.0) * 1.5
    f.set_state(psi)
    f.step_imag(3)
    bad = np.inf if what == "inf" else np.nan
    psi[1, 5, 40] = bad
    if what == "two":
        psi[1, 5, 41] = bad
    s.set_state(psi)
    s.step_imag(3)
    got, ref = s.get_state()[:, 60:], f.get_state()[:, 60:]
    assert not np.any(np.isnan(got))
    assert np.linalg.norm(got - ref) <= 1e-15 * np.linalg.norm(ref)
