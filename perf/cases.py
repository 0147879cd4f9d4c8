"""The work a user of this package has the GPU do, as cases that can be timed and checked.

A pass is what a program does between two looks at its state: put a state on the grid, advance it by a
run of split steps (imaginary time towards a ground state, real time after a quench or under a drive
Omega(t)), and read the observables; or one differentiated propagation. The kinds:

  run      one grid: Solver.load_state, step_imag / step_real, energy_array; the state stays on the GPU
  batch    many uneven grids together: BatchSolver.load_state, step_imag, energy
  adjoint  propagate_real and its backward pass for a cotangent of the final state: the final state and
           the gradients with respect to psi_0, Omega(t) and the trap frequencies

Sizes and parameters are those of bench.py (256, 256 x 256, 512 x 512, 2048 x 2048, the 64-instance
batch, the 256 x 256 gradient), of the tests (640 and 161 x 161 of the paper's Fig. 4, the small uneven
grids) and ragged ones between them. Complex64 runs report their observables and gradients in float32,
the accuracy that form has.

exact() restates the method of arXiv:2009.13507 (Sec. 2, Sec. 3, Appendix A) in plain torch float64.
"""
import math

import numpy as np
import torch

from paper_2009_13507_gb300 import sgpe

DEV = "cuda:0"
RDTYPE = {"c64": torch.float32, "c128": torch.float64, "cdf": torch.float64}
CDTYPE = {"c64": torch.complex64, "c128": torch.complex128, "cdf": torch.complex128}


def _run(name, dim, nx, ny, prec, mode, steps, dx, dt, c0, c2, so_type, gamma, omega, table=False, width=1.0,
         renorm=1, mag=0.0, split=0, so_mode=0):
    return dict(name=name, kind="run", dim=dim, nx=nx, ny=ny, prec=prec, mode=mode, steps=steps, dx=dx, dt=dt, c0=c0,
                c2=c2, so_type=so_type, gamma=gamma, omega=omega, table=table, width=width,
                renorm=renorm if mode == "imag" else 0, mag=mag, split=split, so_mode=so_mode)


def listed():
    return [
        # the smallest grids, a few steps between two looks at the energy: launches and latency count
        _run("small_2d_48x40_c128_imag", 2, 48, 40, "c128", "imag", 10, 0.2, 2e-3, 30.0, 2.0, 2, 0.4, 0.1),
        # the 1D ground state search of the plain form
        _run("1d_256_c128_imag", 1, 256, 1, "c128", "imag", 500, 0.05, 1e-4, 10.0, -0.5, 1, 0.5, 0.2),
        # a long ragged 1D line driven by Omega(t) in the precision form
        _run("1d_1000_c64_real_table", 1, 1000, 1, "c64", "real", 200, 0.04, 1e-4, 60.0, 0.7, 3, 0.9, 0.6,
             table=True, width=4.0),
        # the headline workload: 2D ground state, plain form
        _run("2d_256_c128_imag", 2, 256, 256, "c128", "imag", 50, 0.05, 2e-4, 50.0, 1.0, 1, 0.8, 0.5),
        # the paper's own odd grid in real time after a quench of c0 (Fig. 4), FP64-accurate
        _run("2d_161_c128_real_table", 2, 161, 161, "c128", "real", 50, 0.1, 2.5e-4, 500.0, 15.0, 1, 0.5, 0.3,
             table=True, width=3.0),
        # the same run with the unitary spin-orbit substep and the symmetric splitting
        _run("2d_161_c128_real_strang_socn", 2, 161, 161, "c128", "real", 20, 0.1, 2.5e-4, 500.0, 15.0, 1, 0.5, 0.0,
             width=3.0, split=1, so_mode=1),
        # the double-float form on a ragged mid-size grid
        _run("2d_400x330_cdf_imag", 2, 400, 330, "cdf", "imag", 32, 0.05, 2e-4, 50.0, 1.0, 2, 0.6, 0.5, width=2.0),
        # the headline workload in the precision form
        _run("2d_256_c64_imag", 2, 256, 256, "c64", "imag", 100, 0.05, 2e-4, 50.0, 1.0, 1, 0.8, 0.5),
        # the real-time quench Omega 0.5 -> 0 in the precision form
        _run("2d_512_c64_real", 2, 512, 512, "c64", "real", 200, 0.04, 1e-4, 50.0, 1.0, 1, 0.8, 0.0, width=2.0),
        # a state that no longer fits the L2 cache
        _run("2d_2048_c64_imag", 2, 2048, 2048, "c64", "imag", 100, 0.05, 2e-4, 50.0, 1.0, 1, 0.8, 0.5, width=4.0),
        # 32 1D and 32 2D instances of uneven size and physics
        dict(name="batch_64_c64_imag", kind="batch", n1d=32, n2d=32, lo1=128, hi1=1024, lo2=128, hi2=384, prec="c64",
             steps=50, table_seed=0),
        # the gradient of a driven propagation
        dict(name="adjoint_256_c64", kind="adjoint", dim=2, nx=256, ny=256, prec="c64", steps=100, every=50, dx=0.05,
             dt=2e-4, c0=50.0, c2=1.0, so_type=1, gamma=0.8, omega=0.5, width=1.0),
    ]


# Rough seconds per point-step and per step, only to keep a drawn case below the largest listed one.
_PER_POINT = {"c64": 1.4e-10, "cdf": 3.2e-10, "c128": 7.2e-10}
_CAP_S = 9e-3


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["1d", "2d", "variant", "batch", "adjoint"], [22, 48, 8, 10, 12])[0]
    prec = rng.choices(["c128", "c64", "cdf"], [40, 42, 18])[0]
    # dt = f dx^2: the paper's imaginary and real time steps and bench.py's lie at f = 0.025 .. 0.1
    dx = rng.choice([0.04, 0.05, 0.05, 0.1, 0.2])
    f = rng.choice([0.025, 0.05, 0.08, 0.1, 0.1, 0.4])
    dt = f * dx * dx
    phys = dict(dx=dx, dt=dt, c0=rng.uniform(1.0, 100.0), c2=rng.uniform(-2.0, 2.0), gamma=rng.uniform(0.1, 1.0),
                omega=rng.choice([0.0, rng.uniform(0.0, 1.0)]))
    mode = rng.choice(["imag", "imag", "real"])
    if kind == "batch":
        lo2 = rng.randint(40, 160)
        return dict(kind="batch", n1d=rng.randint(4, 24), n2d=rng.randint(4, 20), lo1=rng.randint(60, 300), hi1=1024,
                    lo2=lo2, hi2=lo2 + rng.randint(10, 120), prec="c64" if prec != "c128" else "c128", steps=rng.randint(8, 20),
                    table_seed=rng.randint(1, 10 ** 6))
    if kind == "1d":
        nx = _logint(rng, 33, 3000)
        width = min(max(0.06 * nx * dx, 0.4), 6.0)
        renorm, mag, so = (2, rng.uniform(-0.5, 0.5), 0) if rng.random() < 0.12 else (1, 0.0, rng.randint(1, 3))
        return _run("", 1, nx, 1, prec, mode, rng.randint(60, 300), so_type=so, table=mode == "real" and rng.random() < 0.5,
                    width=width, renorm=renorm, mag=mag, **phys)
    nx = _logint(rng, 33, 1400)
    ny = min(1400, max(33, int(nx * rng.uniform(0.6, 1.6))))
    if kind in ("variant", "adjoint"):
        nx, ny = min(nx, 300), min(ny, 300)
    if rng.random() < 0.4:
        nx -= nx % 2
    cost = nx * ny * _PER_POINT[prec] + 8e-6
    width = min(max(0.07 * min(nx, ny) * dx, 0.4), 6.0)
    so = rng.randint(1, 3) if rng.random() < 0.85 else 0
    if kind == "adjoint":
        prec = "c64" if prec != "c128" else "c128"
        cost = 9 * (nx * ny * _PER_POINT[prec] + 6e-6)
        steps = max(6, min(rng.randint(20, 60), int(_CAP_S / cost)))
        return dict(kind="adjoint", dim=2, nx=nx, ny=ny, prec=prec, steps=steps, every=rng.choice([5, 8, 20, 50]),
                    so_type=so, width=width, **phys)
    if kind == "variant":
        split, so_mode = rng.choice([(0, 1), (1, 0), (1, 1)])
        steps = max(4, min(rng.randint(10, 40), int(_CAP_S / (4 * cost))))
        return _run("", 2, nx, ny, prec, mode, steps, so_type=max(so, 1), width=width, split=split, so_mode=so_mode, **phys)
    steps = max(4, min(rng.randint(20, 150), int(_CAP_S / cost)))
    renorm, mag, so = (2, rng.uniform(-0.5, 0.5), 0) if rng.random() < 0.1 else (1, 0.0, so)
    return _run("", 2, nx, ny, prec, mode, steps, so_type=so, table=mode == "real" and rng.random() < 0.5, width=width,
                renorm=renorm, mag=mag, **phys)


# -- inputs ------------------------------------------------------------------------------------------------------------
def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFFFFFFFFFF)
    return g


def _gaussian(c, g):
    """[3][ny][nx] complex128: displaced Gaussians of unequal width with a phase gradient, a phase per component
    and a part in a thousand of noise; unit norm."""
    r = torch.rand(24, generator=g, device=DEV, dtype=torch.float64)
    x = ((torch.arange(c["nx"], device=DEV, dtype=torch.float64) - c["nx"] // 2) * c["dx"])[None, None, :]
    y = ((torch.arange(c["ny"], device=DEV, dtype=torch.float64) - c["ny"] // 2) * c["dx"])[None, :, None] if c["dim"] == 2 \
        else torch.zeros(1, 1, 1, device=DEV, dtype=torch.float64)
    w = c["width"] * (0.85 + 0.3 * r[0:3])[:, None, None]
    x0, y0 = 0.3 * w * (r[3:6] - 0.5)[:, None, None], 0.3 * w * (r[6:9] - 0.5)[:, None, None]
    amp = (0.5 + r[9:12])[:, None, None]
    k = (r[12:15] - 0.5)[:, None, None]
    phase = 2 * math.pi * r[15:18][:, None, None] + k * x
    if c["dim"] == 1:
        y0 = y0 * 0
    psi = amp * torch.exp(-((x - x0) ** 2 + (y - y0) ** 2) / (2 * w * w)) * torch.exp(1j * phase)
    u = torch.rand((2, 3, c["ny"], c["nx"]), generator=g, device=DEV, dtype=torch.float64) * 2 - 1
    psi = psi * (1.0 + 1e-3 * torch.complex(u[0], u[1]))
    cell = c["dx"] ** c["dim"]
    return psi / torch.sqrt((psi.abs() ** 2).sum() * cell)


def _omega_table(c, g):
    """A smooth drive around the constant Omega, one value a step."""
    r = torch.rand(3, generator=g, device=DEV, dtype=torch.float64)
    t = torch.arange(c["steps"], device=DEV, dtype=torch.float64) / max(c["steps"], 2)
    return (c["omega"] + 0.3 * r[0] * torch.sin(2 * math.pi * (t * (1 + 2 * r[1]) + r[2]))).contiguous()


def _instances(c):
    rng = np.random.RandomState(c["table_seed"])
    out = []
    for i in range(c["n1d"] + c["n2d"]):
        d1 = i < c["n1d"]
        n = int(rng.randint(c["lo1"], c["hi1"] + 1) if d1 else rng.randint(c["lo2"], c["hi2"] + 1))
        out.append(dict(dim=1 if d1 else 2, nx=n, ny=1 if d1 else n, dx=0.05, dy=0.05, so_type=1, dt=1e-4 if d1 else 2e-4,
                        renorm=1, gamma=float(rng.uniform(0, 1)), omega=float(rng.uniform(0, 1)),
                        c0=float(rng.uniform(1, 100)), c2=float(rng.uniform(-2, 2))))
    return out


def _instance_state(d, g):
    return _gaussian(dict(d, width=1.0), g)


def _physics(c, **kw):
    keys = ("c0", "c2", "so_type", "gamma", "omega", "dt", "renorm", "mag", "split", "so_mode")
    return sgpe.Physics(**dict({k: c[k] for k in keys if k in c}, **kw))


def _inputs(c, seed):
    """The inputs of a case on the GPU, from the seed alone."""
    g = _gen(seed)
    if c["kind"] == "batch":
        return {"psi0": [_instance_state(d, g) for d in _instances(c)]}
    rdt, cdt = RDTYPE[c["prec"]], CDTYPE[c["prec"]]
    psi0 = _gaussian(c, g).to(cdt)
    if c["kind"] == "adjoint":
        cot = _gaussian(c, g).to(cdt)
        w = (1.0 + 0.1 * torch.rand(2, generator=g, device=DEV, dtype=torch.float64)).to(rdt).cpu()
        return {"psi0": psi0, "omega": _omega_table(c, g).to(rdt), "w": w, "cot": cot}
    return {"psi0": psi0, "omega": _omega_table(c, g) if c["table"] else None}


def prepare(case, seed):
    c = case
    st = {"case": c, "in": _inputs(c, seed)}
    torch.cuda.synchronize()  # a solver works on a stream of its own: the inputs are ready before it is made
    if c["kind"] == "batch":
        bs = sgpe.BatchSolver(_instances(c), precision=c["prec"], device=DEV)
        packed = torch.zeros_like(bs.psi)
        for off, p in zip(bs.offsets, st["in"].pop("psi0")):
            packed[off:off + p.numel()] = p.reshape(-1).to(packed.dtype)
        st.update(batch=bs, packed=packed)
        return st
    s = sgpe.Solver(c["dim"], c["nx"], c["ny"], dx=c["dx"], precision=c["prec"], device=DEV)
    if c["kind"] == "adjoint":
        s.set_params(_physics(c, renorm=0))
        i = st["in"]
        for k in ("psi0", "omega", "w"):
            i[k] = i[k].clone().requires_grad_(True)
    else:
        s.set_params(_physics(c))
    st["solver"] = s
    return st


def run(state):
    c, i = state["case"], state["in"]
    if c["kind"] == "batch":
        bs = state["batch"]
        bs.load_state(state["packed"])
        bs.step_imag(c["steps"])
        obs = bs.energy()
        return {"psi": bs.psi, "obs": obs.astype(np.float32) if c["prec"] == "c64" else obs}
    s = state["solver"]
    if c["kind"] == "adjoint":
        psi = sgpe.propagate_real(i["psi0"], i["omega"], i["w"], s, c["every"])
        g = torch.autograd.grad(psi, (i["psi0"], i["omega"], i["w"]), grad_outputs=i["cot"])
        return {"psi": psi.detach(), "dpsi0": g[0], "domega": g[1], "dw": g[2]}
    s.load_state(i["psi0"])
    if c["mode"] == "imag":
        s.step_imag(c["steps"])
    else:
        s.step_real(c["steps"], i["omega"])
    obs = s.energy_array()
    if c["prec"] == "cdf":  # the bound state holds (re_hi, re_lo, im_hi, im_lo)
        p = s.psi.double()
        return {"psi": torch.complex(p[..., 0] + p[..., 1], p[..., 2] + p[..., 3]), "obs": obs}
    return {"psi": s.psi, "obs": obs.astype(np.float32) if c["prec"] == "c64" else obs}


# -- the work of a pass -----------------------------------------------------------------------------------------------
_ESZ = {"c64": 8, "c128": 16, "cdf": 16}
# flops per point and step: the pointwise substeps and one Crank-Nicolson sweep (three components)
_PW = {"imag": 260, "real": 290}
_CN = {"imag": 66, "real": 114}


def work(case):
    c = case
    if c["kind"] == "batch":
        pts = sum(d["nx"] * d["ny"] for d in _instances(c))
        sweeps = sum(d["nx"] * d["ny"] * d["dim"] for d in _instances(c))
        return {"bytes": 2.0 * 3 * pts * _ESZ[c["prec"]],
                "flops": float(c["steps"]) * (pts * (_PW["imag"] + 12) + sweeps * _CN["imag"])}
    pts = c["nx"] * c["ny"]
    state = 3.0 * pts * _ESZ[c["prec"]]
    if c["kind"] == "adjoint":
        # forward, and a reverse of about twice its arithmetic
        return {"bytes": 4 * state + 16.0 * c["steps"], "flops": 3.0 * c["steps"] * pts * (_PW["real"] + 2 * _CN["real"])}
    per = _PW[c["mode"]] * (2 if c["split"] else 1) + c["dim"] * _CN[c["mode"]]
    if c["so_mode"]:
        per += (2 if c["split"] else 1) * c["dim"] * 90
    return {"bytes": 2 * state + (8.0 * c["steps"] if c["table"] else 0.0), "flops": float(c["steps"]) * pts * (per + 12)}


# -- the method in 64 bits ---------------------------------------------------------------------------------------------
def _cn_matrix(n, h, z):
    """(I - z/(4h^2) L)^-1 (I + z/(4h^2) L), L = tridiag(1, -2, 1)."""
    L = -2 * torch.eye(n, dtype=torch.float64, device=DEV)
    L += torch.diag(torch.ones(n - 1, dtype=torch.float64, device=DEV), 1)
    L += torch.diag(torch.ones(n - 1, dtype=torch.float64, device=DEV), -1)
    eye = torch.eye(n, dtype=torch.float64, device=DEV)
    b = z / (4 * h * h)
    if isinstance(z, complex):
        L, eye = L.to(torch.complex128), eye.to(torch.complex128)
    return torch.linalg.solve(eye - b * L, eye + b * L)


def _sweep(M, psi, axis):
    """M applied to every line of psi along axis (-1: x, -2: y)."""
    def mul(a):
        return a @ M.transpose(0, 1) if axis == -1 else torch.matmul(M, a)
    if M.is_complex():
        return mul(psi)
    return torch.complex(mul(psi.real.contiguous()), mul(psi.imag.contiguous()))


def _sweep_sine(n, h, z, psi, axis):
    """The same by the sine transform that diagonalises L (long lines)."""
    k = torch.arange(1, n + 1, dtype=torch.float64, device=DEV)
    lam = 4 * z / (4 * h * h) * torch.sin(math.pi * k / (2 * (n + 1))) ** 2
    f = (1 - lam) / (1 + lam)
    a = psi.transpose(-1, axis)

    def dst(v):
        zero = torch.zeros_like(v[..., :1])
        return torch.fft.fft(torch.cat([zero, v, zero, -v.flip(-1)], -1), dim=-1)[..., 1:n + 1]
    out = torch.empty_like(a)
    for j in range(a.shape[0]):
        out[j] = dst(dst(a[j]) * f) * (-1.0 / (2 * (n + 1)))
    return out.transpose(-1, axis)


def _d(u, axis):
    """psi(+1) - psi(-1) along an axis, zero outside."""
    zero = torch.zeros_like(u.narrow(axis, 0, 1))
    n = u.shape[axis]
    return torch.cat([u.narrow(axis, 1, n - 1), zero], axis) - torch.cat([zero, u.narrow(axis, 0, n - 1)], axis)


def _eta(c):
    return {1: 1.0, 2: -1.0, 3: 0.0}[c["so_type"]]


def _hso(c, psi):
    """H_SO psi."""
    if not c["so_type"] or c["gamma"] == 0.0:
        return torch.zeros_like(psi)
    gt = c["gamma"] / math.sqrt(2.0)
    X = _d(psi, -1) / (2 * c["dx"])
    if c["dim"] == 2:
        Y = _d(psi, -2) / (2 * c["dx"])
        e = _eta(c)
        return torch.stack([gt * X[1] - 1j * gt * e * Y[1], -gt * X[0] + gt * X[2] - 1j * gt * e * (Y[0] + Y[2]),
                            -gt * X[1] - 1j * gt * e * Y[1]])
    if c["so_type"] == 1:
        return torch.stack([-1j * gt * X[1], -1j * gt * (X[0] + X[2]), -1j * gt * X[1]])
    if c["so_type"] == 2:
        return torch.stack([-gt * X[1], gt * (X[0] - X[2]), gt * X[1]])
    return torch.stack([-1j * c["gamma"] * X[0], torch.zeros_like(X[1]), 1j * c["gamma"] * X[2]])


def _so_cayley(c, z, axis):
    """(I + z/2 H)^-1 (I - z/2 H) of the part of H_SO along one axis, on [3 n] lines (2D)."""
    n = c["nx"] if axis == -1 else c["ny"]
    D = (torch.diag(torch.ones(n - 1, dtype=torch.float64, device=DEV), 1)
         - torch.diag(torch.ones(n - 1, dtype=torch.float64, device=DEV), -1)).to(torch.complex128) / (2 * c["dx"])
    gt = c["gamma"] / math.sqrt(2.0)
    if axis == -1:
        S = gt * torch.tensor([[0, 1, 0], [-1, 0, 1], [0, -1, 0]], dtype=torch.complex128, device=DEV)
    else:
        S = -1j * gt * _eta(c) * torch.tensor([[0, 1, 0], [1, 0, 1], [0, 1, 0]], dtype=torch.complex128, device=DEV)
    H = torch.kron(S, D)
    eye = torch.eye(3 * n, dtype=torch.complex128, device=DEV)
    return torch.linalg.solve(eye + z / 2 * H, eye - z / 2 * H)


def _so_cn(c, psi, M, axis):
    p = psi if axis == -1 else psi.transpose(-1, -2)
    q = p.permute(1, 0, 2).reshape(p.shape[1], -1) @ M.transpose(0, 1)
    q = q.reshape(p.shape[1], 3, p.shape[2]).permute(1, 0, 2)
    return q if axis == -1 else q.transpose(-1, -2)


def _potential(c, wx, wy):
    x = (torch.arange(c["nx"], device=DEV, dtype=torch.float64) - c["nx"] // 2) * c["dx"]
    V = 0.5 * wx * wx * x[None, :] ** 2
    if c["dim"] == 2:
        y = (torch.arange(c["ny"], device=DEV, dtype=torch.float64) - c["ny"] // 2) * c["dx"]
        V = V + 0.5 * wy * wy * y[:, None] ** 2
    return V


def _calcnu(c, psi, V, z):
    r = psi.real ** 2 + psi.imag ** 2
    base = V + c["c0"] * (r[0] + r[1] + r[2])
    mu = torch.stack([base + c["c2"] * (r[0] - r[2] + r[1]), base + c["c2"] * (r[0] + r[2]),
                      base + c["c2"] * (r[2] - r[0] + r[1])])
    if isinstance(z, complex):
        return psi * torch.complex(torch.cos(z.imag * mu), -torch.sin(z.imag * mu))
    return psi * torch.exp(-z * mu)


def _herm(c, psi, ot, z):
    """exp(-z A) psi, A = [[0, a, 0], [a*, 0, b], [0, b*, 0]]: A^3 = C^2 A, the series of sinh and cosh in (z C)^2."""
    p, q, m = psi[0], psi[1], psi[2]
    a, b = c["c2"] * m.conj() * q + ot, c["c2"] * q.conj() * p + ot
    C2 = a.real ** 2 + a.imag ** 2 + b.real ** 2 + b.imag ** 2
    v = (z * z).real * C2
    s, k = torch.zeros_like(v), torch.zeros_like(v)
    for n in range(9, -1, -1):
        s = s * v + 1.0 / math.factorial(2 * n + 1)
        k = k * v + 1.0 / math.factorial(2 * n + 2)
    def A(u):
        return torch.stack([a * u[1], a.conj() * u[0] + b * u[2], b.conj() * u[1]])
    A1 = A(psi)
    return psi - z * s * A1 + (z * z).real * k * A(A1)


def _scale(c, psi, cell):
    """The renormalisation factors of Eqs. (DJ2) and (DJ)."""
    if not c.get("renorm", 0):
        return psi
    N = (psi.real ** 2 + psi.imag ** 2).sum((-1, -2)) * cell
    if c["renorm"] == 1:
        return psi / torch.sqrt(N.sum())
    m = c["mag"]
    d0 = math.sqrt(1 - m * m) / torch.sqrt(N[1] + torch.sqrt(4 * (1 - m * m) * N[0] * N[2] + m * m * N[1] ** 2))
    dp = torch.sqrt(1 + m - d0 ** 2 * N[1]) / torch.sqrt(2 * N[0])
    dm = torch.sqrt(1 - m - d0 ** 2 * N[1]) / torch.sqrt(2 * N[2])
    return psi * torch.stack([dp, d0, dm])[:, None, None]


def _propagate(c, psi, imag, steps, omega=None, wx=1.0, wy=1.0):
    dim, cell, dt = c["dim"], c["dx"] ** c["dim"], c["dt"]
    z = dt if imag else 1j * dt
    axes = [(-1, c["nx"])] + ([(-2, c["ny"])] if dim == 2 else [])
    mats = {ax: _cn_matrix(n, c["dx"], z) for ax, n in axes if n <= 1024}
    strang, so_cn = c.get("split", 0), c.get("so_mode", 0) and c["so_type"] and c["gamma"] != 0.0
    zs = z / 2 if strang else z
    cay = [(ax, _so_cayley(c, zs, ax)) for ax, _n in axes if ax == -1 or _eta(c) != 0.0] if so_cn else []
    V = _potential(c, wx, wy)

    def so(p, reverse=False):
        if not so_cn:
            return p - zs * _hso(c, p)
        for ax, M in (reversed(cay) if reverse else cay):
            p = _so_cn(c, p, M, ax)
        return p
    for n in range(steps):
        ot = (c["omega"] if omega is None else omega[n]) / math.sqrt(2.0)
        psi = _herm(c, _calcnu(c, so(psi), V, zs), ot, zs)
        for ax, m in axes:
            psi = _sweep(mats[ax], psi, ax) if ax in mats else _sweep_sine(m, c["dx"], z, psi, ax)
        if strang:
            psi = so(_calcnu(c, _herm(c, psi, ot, zs), V, zs), reverse=True)
        if imag:
            psi = _scale(c, psi, cell)
    return psi


def _observables(c, psi):
    """N_j, N, m, E, mu, rms sizes and the parts of E (the discrete sums on the grid), as energy_array orders them."""
    dim, h, cell = c["dim"], c["dx"], c["dx"] ** c["dim"]
    r = psi.real ** 2 + psi.imag ** 2
    x = (torch.arange(c["nx"], device=DEV, dtype=torch.float64) - c["nx"] // 2) * h
    rr = x[None, :] ** 2
    if dim == 2:
        rr = rr + ((torch.arange(c["ny"], device=DEV, dtype=torch.float64) - c["ny"] // 2) * h)[:, None] ** 2
    kin = 0.0
    for ax in ((-1, -2) if dim == 2 else (-1,)):
        zero = torch.zeros_like(psi.narrow(ax, 0, 1))
        d = torch.cat([psi, zero], ax) - torch.cat([zero, psi], ax)
        kin = kin + 0.5 * (d.real ** 2 + d.imag ** 2).sum() / (h * h) * cell
    N = r.sum((-1, -2)) * cell
    rho = r.sum(0)
    trap = (_potential(c, 1.0, 1.0) * rho).sum() * cell
    x4 = (psi[2].conj() * psi[1] ** 2 * psi[0].conj()).real
    inter = 0.5 * (c["c0"] * rho ** 2 + c["c2"] * (r[0] ** 2 + r[2] ** 2 + 2 * r[0] * r[1] + 2 * r[2] * r[1]
                                                     - 2 * r[0] * r[2] + 4 * x4)).sum() * cell
    rabi = 2 * c["omega"] / math.sqrt(2.0) * ((psi[0] + psi[2]).conj() * psi[1]).real.sum() * cell
    so = (psi.conj() * _hso(c, psi)).real.sum() * cell
    rj = (rr * r).sum((-1, -2)) * cell
    E, Nt = kin + trap + inter + rabi + so, N.sum()
    v = [N[0], N[1], N[2], Nt, N[0] - N[2], E, (kin + trap + so + rabi + 2 * inter) / Nt, torch.sqrt(rj[0] / N[0]),
         torch.sqrt(rj[1] / N[1]), torch.sqrt(rj[2] / N[2]), torch.sqrt(rj.sum() / Nt), kin, trap, inter, rabi, so]
    return torch.stack([t.to(torch.float64) for t in v])


def exact(case, seed):
    c, i = case, _inputs(case, seed)
    if c["kind"] == "batch":
        insts = _instances(c)
        cdt = CDTYPE[c["prec"]]
        parts, obs = [], []
        for d, p0 in zip(insts, i["psi0"]):
            p = _propagate(d, p0.to(cdt).to(torch.complex128), True, c["steps"])
            obs.append(_observables(d, p))
            parts.append(p.reshape(-1))
        # the states follow one another, each from a multiple of 64 elements
        parts = [torch.nn.functional.pad(p, (0, -p.numel() % 64)) for p in parts]
        return {"psi": torch.cat(parts), "obs": torch.stack(obs)}
    if c["kind"] == "adjoint":
        psi0 = i["psi0"].to(torch.complex128).requires_grad_(True)
        om = i["omega"].to(torch.float64).requires_grad_(True)
        w = i["w"].to(torch.float64).to(DEV).requires_grad_(True)
        psi = _propagate(c, psi0, False, c["steps"], om, w[0], w[1])
        g = torch.autograd.grad(psi, (psi0, om, w), grad_outputs=i["cot"].to(torch.complex128))
        return {"psi": psi.detach(), "dpsi0": g[0], "domega": g[1], "dw": g[2]}
    psi = _propagate(c, i["psi0"].to(torch.complex128), c["mode"] == "imag", c["steps"], i["omega"])
    return {"psi": psi, "obs": _observables(c, psi)}
