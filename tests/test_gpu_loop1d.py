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


@pytest.mark.parametrize("precision", ["c128", "c64"])
@pytest.mark.parametrize("renorm", [1, 2])
def test_more_lines_than_sms_in_a_batch(precision, renorm):
    """Batches with more lines of 129..512 points than SMs run two lines an SM: the first, a middle
    and the last line of each length against the oracle, both time modes."""
    import torch
    from paper_2009_13507_gb300 import sgpe
    count = torch.cuda.get_device_properties(0).multi_processor_count + 8
    lens = [129 + i % 100 for i in range(count)] + [257 + i % 250 for i in range(count)] + [40]
    phys = dict(c0=15.0, c2=-0.5, so_type=0 if renorm == 2 else 1, gamma=0.4, omega=0.2, dt=1e-3, renorm=renorm,
                mag=0.1 if renorm == 2 else 0.0)
    bs = sgpe.BatchSolver([dict(dim=1, nx=n, dx=0.1, **phys) for n in lens], precision=precision)
    states = [I.gaussian_jitter_1d(n, 0.1, seed=n, amp=1e-2) for n in lens]
    bs.load_state(bs.pack(states))
    bs.step_imag(10)
    bs.step_real(3)
    got = bs.states()
    for i in (0, count // 2, count - 1, count, count + count // 2, 2 * count - 1, 2 * count):
        prob = O.Problem(dim=1, nx=lens[i], ny=1, dx=0.1, dy=0.1, **phys)
        ref = O.step(prob, O.step(prob, states[i], 10, True), 3, False)
        assert relerr(got[i], ref) < (1e-10 if precision == "c128" else 1e-5), lens[i]
