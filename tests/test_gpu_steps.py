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


@pytest.mark.parametrize("precision", ["c128", "c64", "cdf"])
@pytest.mark.parametrize("dim,nx,ny,so", [(2, 32, 5, 1), (2, 33, 9, 2), (2, 31, 3, 3), (2, 64, 64, 0), (2, 300, 517, 1),
                                          (1, 128, 1, 1), (1, 129, 1, 2), (1, 97, 1, 3)])
def test_observable_strips(dim, nx, ny, so, precision):
    """Strips that end inside a block, at a warp's last column (the ghost link) or
    before the grid does, every SO term as link sums, and complex64 values that
    underflow to zero or subnormals. The sums are FP64 over the state as it is
    stored: 1e-12 of the largest observable (about 100 roundings of the largest sum)."""
    prob, s = make_pair(dim, nx, ny, dx=0.2, dy=0.25 if dim == 2 else None, c0=30.0, c2=-1.5, so_type=so, gamma=0.7,
                        omega=0.4, wx=1.0, wy=1.2, dt=1e-3, precision=precision)
    psi = _rand(prob, 40 + nx, env=60.0)
    psi[2] *= 1e-30  # complex64: subnormals where the envelope is small
    psi[:, :, : nx // 4] = 0.0
    if precision == "c64":
        psi = psi.astype(np.complex64).astype(np.complex128)
    s.set_state(psi)
    got, ref = s.energy_array(), O.observables_array(prob, psi)
    keep = [i for i in range(16) if i != 9]  # the rms size of a component of norm 1e-60 is 0/0 in float32
    assert np.max(np.abs(got - ref)[keep]) < 1e-12 * np.max(np.abs(ref))


@pytest.mark.parametrize("imag", [True, False])
@pytest.mark.parametrize("nx,ny", [(129, 130), (257, 140), (511, 129), (1025, 36), (1501, 33)])
def test_odd_rows_in_the_fused_row_kernel(nx, ny, imag):
    """complex64 grids with odd rows: 8-byte loads, the last pair's second point past
    the row, zero ghosts there. The bound is the precision form's 1e-5."""
    prob, s = make_pair(2, nx, ny, dx=0.05, c0=40.0, c2=1.0, so_type=1, gamma=0.8, omega=0.5, dt=2e-4,
                        renorm=1 if imag else 0, precision="c64")
    psi = _rand(prob, nx)
    s.set_state(psi)
    (s.step_imag if imag else s.step_real)(12)
    assert relerr(s.get_state(), O.step(prob, psi, 12, imag)) < 1e-5


@pytest.mark.parametrize("precision", ["c128", "c64"])
def test_batch_of_lines_only(precision):
    """1D instances in their step loops: every chunk length from 1 to 32 points a
    lane, the shortest and longest lines, a graph of 32 steps and the rest, both
    time modes."""
    from paper_2009_13507_gb300 import sgpe
    lens = [3, 32, 33, 100, 128, 129, 300, 513, 1024]
    phys = [dict(c0=5.0 + i, c2=-0.5 + 0.1 * i, so_type=1 + i % 3, gamma=0.5, omega=0.2, dt=2e-3, renorm=1)
            for i in range(len(lens))]
    bs = sgpe.BatchSolver([dict(dim=1, nx=n, dx=0.1, **p) for n, p in zip(lens, phys)], precision=precision)
    states = [I.gaussian_jitter_1d(n, 0.1, seed=n, amp=1e-2) for n in lens]
    bs.load_state(bs.pack(states))
    bs.step_imag(40)
    bs.step_real(5)
    obs = bs.energy()
    for i, (n, p) in enumerate(zip(lens, phys)):
        prob = O.Problem(dim=1, nx=n, ny=1, dx=0.1, dy=0.1, **p)
        ref = O.step(prob, O.step(prob, states[i], 40, True), 5, False)
        tol = 1e-10 if precision == "c128" else 1e-5
        assert relerr(bs.states()[i], ref) < tol, n
        assert abs(obs[i, 5] - O.observables(prob, ref)["E"]) < tol * max(1.0, abs(obs[i, 5])), n


PAIR_SIZES = [(17, 91), (33, 47), (128, 128), (127, 129), (160, 64), (161, 65), (256, 48), (257, 47), (300, 81), (18, 200)]
# 20 steps of about ten roundings each, of 2^-53 (complex128) or 2^-48 (double-float), all one way
PAIR_TOL = {"c128": 20 * 10 * 2.0 ** -53, "cdf": 20 * 10 * 2.0 ** -48}


@pytest.mark.parametrize("precision", ["c128", "cdf"])
@pytest.mark.parametrize("imag", [True, False])
@pytest.mark.parametrize("nx,ny", PAIR_SIZES)
def test_pair_step(nx, ny, imag, precision):
    """The pair step at the edges of its row segments (160 and 256 points) and tiles (8
    columns, 64 rows), just above the shortest line, with both head kernels."""
    prob, s = make_pair(2, nx, ny, dx=0.1, dy=0.11, c0=40.0, c2=1.5, so_type=1 + nx % 3, gamma=0.7, omega=0.4, wy=1.1,
                        dt=1e-3, renorm=1 if imag else 0, precision=precision)
    psi = _rand(prob, nx + ny, env=20.0)
    s.set_state(psi)
    (s.step_imag if imag else s.step_real)(20)
    assert relerr(s.get_state(), O.step(prob, psi, 20, imag)) < PAIR_TOL[precision]


@pytest.mark.parametrize("nx", [96, 300])
@pytest.mark.parametrize("what", ["large_dt", "magnetisation", "norm", "tiny", "huge", "table"])
def test_pair_step_outside_its_increments(what, nx):
    """Blocks that leave the increments for FP64 (dt mu, dt A above their limits), scale
    factors far from 1 or unequal, states far from order 1 in linear runs, and a table."""
    kw = dict(c0=40.0, c2=1.5, so_type=1, gamma=0.7, omega=0.4, dt=1e-3, renorm=0)
    imag, scale = False, 1.0
    if what == "large_dt":
        kw.update(dt=2.5e-3, omega=30.0)
    elif what in ("magnetisation", "norm"):
        imag, scale = True, 7.0
        kw.update(renorm=2 if what == "magnetisation" else 1, mag=0.2, so_type=0 if what == "magnetisation" else 1)
    elif what in ("tiny", "huge"):
        scale = 1e-80 if what == "tiny" else 1e60
        kw.update(c0=0.0, c2=0.0)
    prob, s = make_pair(2, nx, 70, dx=0.1, **kw)
    psi = _rand(prob, 5, env=20.0) * scale
    s.set_state(psi)
    if what == "table":
        import torch
        om = np.linspace(0.1, 1.5, 20)
        s.step_real(20, torch.from_numpy(om).cuda())
        ref = O.step(prob, psi, 20, False, om)
    else:
        (s.step_imag if imag else s.step_real)(20)
        ref = O.step(prob, psi, 20, imag)
    assert relerr(s.get_state(), ref) < PAIR_TOL["c128"]


def test_pair_step_reports_a_non_finite_state():
    from paper_2009_13507_gb300 import sgpe
    prob, s = make_pair(2, 64, 40, dx=0.1, c0=1.0, so_type=1, gamma=0.3, dt=1e-3)
    psi = _rand(prob, 1)
    psi[1, 20, 30] = np.nan
    s.set_state(psi)
    s.step_imag(3)
    with pytest.raises(sgpe.SgpeError) as e:
        s.energy()
    assert e.value.status == sgpe.ENONFINITE


@pytest.mark.parametrize("imag", [True, False])
@pytest.mark.parametrize("nx,bt", [(17, 0.02), (31, 0.02), (32, 0.3), (33, 0.02), (257, 0.1), (1024, 0.02), (16, 0.02), (64, 0.5)])
def test_1d_complex64_loop(nx, bt, imag):
    """The one-block loop with its convolution sweep: the shortest and longest lines, taps that
    reach across the line's images, and the lines and bt that stay on the lane-chunk loop. The
    bound is the precision form's 1e-5."""
    dx = 0.1
    prob, s = make_pair(1, nx, 1, dx=dx, c0=20.0, c2=-0.8, so_type=1 + nx % 3, gamma=0.5, omega=0.3,
                        dt=4.0 * dx * dx * bt * (1.0 if bt < 0.05 else 0.1), renorm=(2 if nx == 33 else 1) if imag else 0,
                        mag=0.1, precision="c64")
    if bt >= 0.05:  # a larger bt at an affordable dt: a finer grid
        prob, s = make_pair(1, nx, 1, dx=dx / np.sqrt(10.0), c0=20.0, c2=-0.8, so_type=1 + nx % 3, gamma=0.5, omega=0.3,
                            dt=4.0 * dx * dx * bt * 0.1, renorm=1 if imag else 0, precision="c64")
    psi = _rand(prob, nx, env=10.0)
    s.set_state(psi)
    (s.step_imag if imag else s.step_real)(15)
    assert relerr(s.get_state(), O.step(prob, psi, 15, imag)) < 1e-5
    N = s.normalize()
    ref = O.observables(prob, O.step(prob, psi, 15, imag))
    assert np.max(np.abs(N - [ref["N+"], ref["N0"], ref["N-"]])) < 1e-5


@pytest.mark.parametrize("dim,nx,ny,so", [(2, 20, 16, 1), (2, 32, 8, 2), (2, 33, 9, 1), (2, 31, 7, 3), (2, 64, 17, 0),
                                          (2, 5, 3, 1), (1, 48, 1, 2), (1, 33, 1, 1), (1, 32, 1, 3)])
def test_adjoint_tiles_complex64(dim, nx, ny, so):
    """The complex64 reverse stage in tiles of 32 x 8 points: grids of one tile, a tile and a
    point more, partial tiles, a line; odd and even numbers of steps and a last segment of one.
    Against the complex128 gradient of the same inputs. Bounds: psi_0's cotangent passes 2 x 13
    steps of some 30 roundings of 6e-8 (5e-5 if all add up; 1e-4); dL/dOmega and dL/dw cancel
    over the grid (the precision form's 2e-3 of the largest)."""
    import torch
    from paper_2009_13507_gb300 import sgpe
    phys = dict(c0=15.0, c2=-1.5, so_type=so, gamma=0.7, omega=0.5, wx=1.1, wy=0.9, dt=1e-2, renorm=0)
    om = 0.5 + 0.3 * np.sin(np.arange(13) * 0.7)
    grads = {}
    for prec in ("c128", "c64"):
        prob, s = make_pair(dim, nx, ny, dx=0.35, dy=0.4 if dim == 2 else None, precision=prec, **phys)
        psi = _rand(prob, nx + ny, env=3.0)
        target = _rand(prob, 7 + nx, env=3.0)
        p0 = torch.from_numpy(psi).to(s.cdtype).cuda().requires_grad_(True)
        omt = torch.tensor(om, dtype=torch.float64, device="cuda:0", requires_grad=True)
        w = torch.tensor([1.1, 0.9], dtype=torch.float64, device="cuda:0", requires_grad=True)
        out = sgpe.propagate_real(p0, omt, w, s, 4)
        t = torch.from_numpy(target).to(s.cdtype).cuda().reshape(out.shape)
        rho = out.real ** 2 + out.imag ** 2
        ((torch.conj(t) * out).real.sum() + (rho * (t.real ** 2)).sum()).backward()
        grads[prec] = (p0.grad.cpu().numpy().astype(np.complex128), omt.grad.cpu().numpy(), w.grad.cpu().numpy())
    a, b = grads["c64"], grads["c128"]
    assert np.linalg.norm(a[0] - b[0]) < 1e-4 * np.linalg.norm(b[0])
    assert np.max(np.abs(a[1] - b[1])) < 2e-3 * np.max(np.abs(b[1]))
    assert np.max(np.abs(a[2] - b[2])) < 2e-3 * np.max(np.abs(b[2]))


@pytest.mark.parametrize("precision", ["c128", "c64"])
@pytest.mark.parametrize("K", [1, 4, 12, 13, 50])
def test_adjoint_tape_is_reusable(K, precision):
    """The first reverse pass of a tape takes the last segment's states from the forward pass, a
    second one recomputes them (one segment, segments of one step, a last segment of one step, a
    full last one): the same bits, also where loss_grad's own reverse pass used the workspace
    before."""
    import ctypes
    import torch
    prob, s = make_pair(2, 36, 20, dx=0.35, precision=precision, c0=15.0, c2=-1.5, so_type=1, gamma=0.7, omega=0.5, dt=1e-2)
    psi = _rand(prob, 1)
    om = 0.5 + 0.3 * np.sin(np.arange(13) * 0.7)
    lam = torch.from_numpy(_rand(prob, 2)).to(s.cdtype).cuda()
    s.set_state(psi)
    tape = s.adjoint_forward(om, K)
    runs = [s.adjoint_step(tape, lam) for _ in range(2)]
    final = s.get_state()
    s.set_state(psi)
    tgt = torch.zeros(20, 36, dtype=torch.float64, device="cuda:0")
    dom, dw, L = torch.zeros(13, dtype=torch.float64, device="cuda:0"), np.zeros(2), np.zeros(1)
    torch.cuda.synchronize()
    s._check(s.lib.sgpe_adjoint_loss_grad(s.ctx, 13, tape["omega"].data_ptr(), tgt.data_ptr(), K, tape["ws"].data_ptr(),
                                          L.ctypes.data, dom.data_ptr(), dw.ctypes.data))
    runs.append(s.adjoint_step(tape, lam))
    s.synchronize()
    assert np.array_equal(final, s.get_state())
    assert relerr(final, O.step(prob, psi, 13, False, om)) < (1e-11 if precision == "c128" else 1e-5)
    for g, d, w in runs[1:]:
        assert torch.equal(g, runs[0][0]) and torch.equal(d, runs[0][1]) and w == runs[0][2]
