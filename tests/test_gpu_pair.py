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


LD, CL = np.longdouble, np.clongdouble


def _long_sweep(p, b, ax):
    """(I - b L)^-1 (I + b L) p along an axis, L = tridiag(1, -2, 1), in long double."""
    p = np.moveaxis(p, ax, 0)
    d = (1 - 2 * b) * p
    d[1:] += b * p[:-1]
    d[:-1] += b * p[1:]
    c = np.zeros(len(p), CL)
    m = 1 + 2 * b
    c[0], d[0] = -b / m, d[0] / m
    for i in range(1, len(p)):
        m = 1 + 2 * b + b * c[i - 1]
        c[i], d[i] = -b / m, (d[i] + b * d[i - 1]) / m
    for i in range(len(p) - 2, -1, -1):
        d[i] -= c[i] * d[i + 1]
    return np.moveaxis(d, 0, ax)


def _long_steps(psi, steps, imag, dx, dt, c0, c2, gamma, omega):
    """The Lie step with Rashba SO by explicit Euler (renormalised in imaginary time), in long double."""
    psi, dx, dt = psi.astype(CL), LD(dx), LD(dt)
    z = CL(dt) if imag else CL(1j) * dt
    g, ot = LD(gamma) / np.sqrt(LD(2)), LD(omega) / np.sqrt(LD(2))
    ny, nx = psi.shape[1:]
    V = ((((np.arange(nx) - nx // 2) * dx) ** 2)[None, :] + (((np.arange(ny) - ny // 2) * dx) ** 2)[:, None]) / 2

    def diff(u, ax):
        o = np.zeros_like(u)
        a, b = np.moveaxis(u, ax, 0), np.moveaxis(o, ax, 0)
        b[:-1] += a[1:]
        b[1:] -= a[:-1]
        return o / (2 * dx)
    for _ in range(steps):
        X, Y = diff(psi, 2), diff(psi, 1)
        psi = psi - z * g * np.stack([X[1] - 1j * Y[1], X[2] - X[0] - 1j * (Y[0] + Y[2]), -X[1] - 1j * Y[1]])
        r = psi.real ** 2 + psi.imag ** 2
        mu = np.stack([(r[0] - r[2]) + r[1], r[0] + r[2], (r[2] - r[0]) + r[1]]) * LD(c2) + V + LD(c0) * r.sum(0)
        psi = psi * np.exp(-z * mu)
        a, b = c2 * psi[2].conj() * psi[1] + ot, c2 * psi[1].conj() * psi[0] + ot
        v = (z * z).real * (abs(a) ** 2 + abs(b) ** 2)
        s = 1 + v / 6 * (1 + v / 20 * (1 + v / 42 * (1 + v / 72)))
        k = LD(1) / 2 + v / 24 * (1 + v / 30 * (1 + v / 56 * (1 + v / 90)))
        A1 = np.stack([a * psi[1], a.conj() * psi[0] + b * psi[2], b.conj() * psi[1]])
        A2 = np.stack([a * A1[1], a.conj() * A1[0] + b * A1[2], b.conj() * A1[1]])
        psi = psi - z * s * A1 + (z * z).real * k * A2
        for ax in (2, 1):
            psi = _long_sweep(psi, z / (4 * dx * dx), ax)
        if imag:
            psi = psi / np.sqrt((psi.real ** 2 + psi.imag ** 2).sum() * dx * dx)
    return psi


@pytest.mark.parametrize("imag", [True, False])
@pytest.mark.parametrize("nx,ny,steps,dx,dt,gamma", [
    (64, 48, 10, 0.1, 2.5e-3, 0.8), (64, 48, 10, 0.05, 8e-4, 0.8), (64, 48, 10, 0.1, 2.5e-3, 20.0),
    (64, 48, 10, 0.05, 2e-4, 0.8), (168, 100, 5, 0.05, 8e-4, 0.8), (168, 100, 5, 0.1, 2.5e-3, 20.0)])
def test_rough_states_keep_the_accuracy_of_fp64(nx, ny, steps, dx, dt, gamma, imag):
    """Independent random values at every point, bt up to the most taps, strong SO: SO's and the
    sweeps' increments are no longer small and leave the pairs. Against long double; the
    bound is what nine roundings of 2^-53 a step (SO, CALCNU, HERM, two sweeps, the state between
    them) leave when their signs are random: 3 * 2^-53 * sqrt(steps)."""
    if np.finfo(LD).eps > 2.0 ** -60:
        pytest.skip("long double is no wider than double here")
    prob, s = make_pair(2, nx, ny, dx=dx, dt=dt, c0=20.0, c2=1.0, so_type=1, gamma=gamma, omega=0.5, renorm=1 if imag else 0)
    psi = _rand(prob, nx + ny, env=8.0)
    s.set_state(psi)
    (s.step_imag if imag else s.step_real)(steps)
    ref = _long_steps(psi, steps, imag, dx, dt, 20.0, 1.0, gamma, 0.5)
    err = np.sqrt((abs(s.get_state() - ref) ** 2).sum() / (abs(ref) ** 2).sum())
    assert err < 3 * 2.0 ** -53 * np.sqrt(steps)


@pytest.mark.parametrize("imag", [True, False])
@pytest.mark.parametrize("nx,ny", [(64, 48), (168, 100)])
@pytest.mark.parametrize("what", ["herm", "density", "both"])
def test_large_nonlinear_increments(what, nx, ny, imag):
    """dt A between 2^-10 and 2^-6 (the HERM coefficients as a series in pairs), and a dense narrow
    state: blocks whose dt mu sends them to FP64 from the start (its centre), after the vote (its
    flanks) and not at all. Against long double, the bound of the rough states."""
    if np.finfo(LD).eps > 2.0 ** -60:
        pytest.skip("long double is no wider than double here")
    omega, c0 = (0.5 if what == "density" else 7.0), (5.0 if what == "herm" else 60.0)
    dx, dt, steps = 0.05, 8e-4, 8
    prob, s = make_pair(2, nx, ny, dx=dx, dt=dt, c0=c0, c2=1.0, so_type=1, gamma=0.5, omega=omega, renorm=1 if imag else 0)
    x, y = (np.arange(nx) - nx // 2) * dx, (np.arange(ny) - ny // 2) * dx
    psi = np.stack([a * np.exp(-((x[None] - b) ** 2 + y[:, None] ** 2) / 0.32 + 0.3j * x[None]) for a, b in ((1.0, 0.05), (0.9, 0.0), (0.8j, -0.05))])
    psi = psi / np.sqrt((abs(psi) ** 2).sum() * dx * dx)
    s.set_state(psi)
    (s.step_imag if imag else s.step_real)(steps)
    ref = _long_steps(psi, steps, imag, dx, dt, c0, 1.0, 0.5, omega)
    err = np.sqrt((abs(s.get_state() - ref) ** 2).sum() / (abs(ref) ** 2).sum())
    assert err < 3 * 2.0 ** -53 * np.sqrt(steps)


def test_the_slot_of_the_largest_value_stays_a_slot(tmp_path):
    """The step's index into the three slots of the state's largest value counts modulo three: a
    count of steps passes 2^31 within hours and its remainder then indexes in front of the slots."""
    import subprocess

    from paper_2009_13507_gb300 import build as B
    src, exe = tmp_path / "probe.cu", tmp_path / "probe"
    src.write_text('#include <stddef.h>\n#include <stdio.h>\n#include "sgpe_kernels.cuh"\n'
                   'int main() { printf("%zu", offsetof(sgpe::DevScalars, pair_tick)); }\n')
    subprocess.run([B._nvcc(), *B.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", B.CSRC, "-o", str(exe), str(src)],
                   check=True, capture_output=True)
    at = int(subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout)
    _, s = make_pair(2, 64, 48, dx=0.1, c0=1.0, so_type=1, gamma=0.3, dt=1e-3)
    s.set_state(I.random_state((3, 48, 64), 1, 0.01, 20.0))
    for n in (1, 1, 1, 7, 40):
        s.step_imag(n)
        s.synchronize()
        assert 0 <= int(s.workspace[at:at + 4].cpu().numpy().view(np.int32)[0]) < 3


@pytest.mark.parametrize("nx,ny", [(64, 48), (168, 100)])
@pytest.mark.parametrize("what", ["small_norm", "large_norm", "tiny_rough", "huge_rough"])
def test_scales_far_from_one(what, nx, ny):
    """Factors beyond 10^6 in the first renormalised step (the shift starts anew, SO with the factors
    of its sources), and rough states with strong SO far from order 1 in linear real-time runs (blocks
    in FP64 under a shift). Against long double, the bound of the rough states."""
    if np.finfo(LD).eps > 2.0 ** -60:
        pytest.skip("long double is no wider than double here")
    imag = what.endswith("norm")
    scale = {"small_norm": 1e-8, "large_norm": 1e8, "tiny_rough": 1e-80, "huge_rough": 1e60}[what]
    c0 = 40.0 if what == "small_norm" else 0.0
    c2, gamma, dx, dt, steps = (1.0 if c0 else 0.0), (0.8 if imag else 20.0), 0.1, 2e-3, 8
    prob, s = make_pair(2, nx, ny, dx=dx, dt=dt, c0=c0, c2=c2, so_type=1, gamma=gamma, omega=0.5, renorm=1 if imag else 0)
    psi = _rand(prob, 2 * nx + ny, env=8.0) * scale
    s.set_state(psi)
    (s.step_imag if imag else s.step_real)(steps)
    ref = _long_steps(psi, steps, imag, dx, dt, c0, c2, gamma, 0.5)
    err = np.sqrt((abs(s.get_state() / scale - ref / scale) ** 2).sum() / (abs(ref / scale) ** 2).sum())
    assert err < 3 * 2.0 ** -53 * np.sqrt(steps)
