"""What the performance of this framework is measured on: calls of its public
entry points as programs make them, over the sizes of the configurations and
tests of this repository.

Kinds of case:
  step         Grid.step(steps) on a grid whose state lives in the caller's
               device tensors (bind_device_fields): one run of the paper, in
               its coarsening regime, inertial (rho > 0) or Stokes (rho = 0),
               FP32 or FP64.  Returns the state after the steps.
  host         Grid.step_host_f32: the state goes in from pinned host memory and
               comes back to it, for programs that keep the fields on the host.
  ensemble     Ensemble.step(steps), then every member's fields are read: a
               parameter sweep of uneven sizes, shear rates and regimes.
  observables  structure_factor with bins, gradient_tensor and mass of one
               state: what a logged run asks for between its steps.

Sizes are powers of two (the library takes no others); step counts, member
counts, aspect ratios and strains are uneven.
"""
import math

import numpy as np
import torch

import paper_0710_5912_gb300 as shf
from paper_0710_5912_gb300 import configs

UNIT = dict(a=1.0, b=1.0, kappa=1.0, M=1.0, eta=1.0, dx=1.0, dt=0.005)


def _step(name, nx, ny, prec, steps, n0, start="domains", **p):
    c = dict(kind="step", name=name, nx=nx, ny=ny, prec=prec, steps=steps, n0=n0, start=start)
    c.update(UNIT)
    c.update(p)
    return c


def _table(row):
    nx, ny, dx, p = configs.paper_units(row)
    return dict(p, dx=dx, nx=nx, ny=ny)


def listed():
    return [
        # the smallest configuration, a quench of 64^2 points without inertia, 100 steps at a time
        _step("quench_64_stokes_fp64", 64, 64, 64, 100, 0, "quench", rho=0.0, gdot=0.01),
        # one step per call: a program that looks at or changes the state after every step
        _step("call_256_inertial", 256, 256, 32, 1, 2000, rho=1.0, gdot=0.003),
        # a small production run between two log lines
        _step("run_256_inertial", 256, 256, 32, 100, 2000, rho=1.0, gdot=0.003),
        # the paper's sheared runs (Table I) on its 1024 x 512 mesh in its units, the strain wrapping on the way
        _step("sheared_1024x512_inertial", prec=32, steps=100, n0=1600, **_table("R028s")),
        _step("sheared_1024x512_stokes", prec=32, steps=20, n0=900, **_table("DV3s")),
        # the side-by-side runs at 1024^2, with and without inertia
        _step("run_1024_inertial", 1024, 1024, 32, 20, 5000, rho=0.1, gdot=0.003),
        _step("run_1024_stokes", 1024, 1024, 32, 20, 5000, rho=0.0, gdot=0.003),
        # the double-precision path, which the single-precision one is checked against
        _step("run_1024_inertial_fp64", 1024, 1024, 64, 5, 5000, rho=1.0, gdot=0.003),
        # the largest configuration
        _step("run_4096_inertial", 4096, 4096, 32, 10, 20000, rho=1.0, gdot=0.001),
        # the same with host arrays in and out at every step
        dict(_step("host_4096_inertial", 4096, 4096, 32, 1, 20000, rho=1.0, gdot=0.001), kind="host"),
        # a sweep of 24 runs of 128^2, 256^2 and 512^2, half of them without inertia
        dict(kind="ensemble", name="ensemble_24", runs=24, small=128, sizes=3, steps=100, n0=3000),
        # what a logged run measures between its steps
        dict(_step("observables_1024", 1024, 1024, 32, 0, 5000, rho=1.0, gdot=0.003), kind="observables", bins=512),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


MOST_POINT_STEPS = 4096 * 4096 * 10


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["ensemble", "host", "observables", "observables"])
    if kind == "ensemble":
        sizes = rng.randint(1, 4)
        small = 2 ** rng.randint(5, 9 - sizes + 1)
        return dict(kind=kind, runs=rng.randint(2, 24), small=small, sizes=sizes,
                    steps=int(_log_uniform(rng, 10, 120)), n0=rng.randint(0, 20000))
    nx = 2 ** rng.randint(5, 12)
    ny = max(16, nx >> rng.choice([0, 0, 0, 1, 1, 2]))
    prec = 64 if kind in ("step", "observables") and nx <= 1024 and rng.random() < 0.3 else 32
    rho = rng.choice([0.0, 0.0, 0.1, 1.0, _log_uniform(rng, 0.05, 20.0)])
    gdot = rng.choice([1, 1, 1, -1]) * _log_uniform(rng, 1e-4, 3e-2)
    c = _step("", nx, ny, prec, 0, rng.randint(0, 40000), rho=rho, gdot=gdot)
    del c["name"]
    c["kind"] = kind
    if kind == "host":
        c["steps"] = rng.choice([1, 1, 2, 7])
    elif kind == "observables":
        c["bins"] = rng.choice([0, int(_log_uniform(rng, 16, 2048))])
    else:
        cost = nx * ny * (25 if prec == 64 else 1) * (2 if rho == 0.0 else 1)
        c["steps"] = max(1, min(int(_log_uniform(rng, 1, 400)), MOST_POINT_STEPS // cost))
    return c


# ------------------------------------------------------------------- inputs

def _strain(n, gdot, dt, nx, ny):
    r = nx // ny
    total = (gdot * dt) * float(n)
    K = math.floor(total / r + 0.5)
    return total - K * r, K


def _wavenumbers(nx, ny, dx, s, device):
    """qx (1, nx/2 + 1), ky = qy - s qx and k^2 (ny, nx/2 + 1), and the mask of
    the modes off the Nyquist lines."""
    m = torch.arange(nx // 2 + 1, device=device, dtype=torch.float64)[None, :]
    n = torch.arange(ny, device=device, dtype=torch.float64)[:, None]
    n = torch.where(n < ny // 2, n, n - ny)
    qx = 2.0 * math.pi / (nx * dx) * m
    ky = 2.0 * math.pi / (ny * dx) * n - s * qx
    keep = ((m != nx // 2) & (n != -(ny // 2))).to(torch.float64)
    return qx, ky, qx * qx + ky * ky, keep


def _smooth(gen, nx, ny, cells):
    """Gaussian noise smoothed over `cells` points, unit variance, zero mean."""
    f = torch.fft.rfft2(torch.randn((ny, nx), generator=gen, device="cuda", dtype=torch.float64))
    qx, ky, k2, keep = _wavenumbers(nx, ny, 1.0, 0.0, "cuda")
    f = f * torch.exp(-0.25 * k2 * cells * cells) * keep
    f[0, 0] = 0.0
    f = torch.fft.irfft2(f, s=(ny, nx))
    return f / f.std()


def _fields(c, seed):
    """(phi, psi, omega) on the GPU in the case's precision: a quench (noise of
    amplitude 0.01 at rest), or domains of phi near +-1 with interfaces of a few
    points and a smooth flow at a tenth of the capillary velocity."""
    nx, ny, dt = c["nx"], c["ny"], torch.float64 if c["prec"] == 64 else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    if c["start"] == "quench":
        phi = 0.01 * (2.0 * torch.rand((ny, nx), generator=gen, device="cuda", dtype=torch.float64) - 1.0)
        psi = torch.zeros_like(phi)
        return phi.to(dt), psi.to(dt), torch.zeros_like(psi).to(dt)
    cells = min(12.0, nx / 8.0, ny / 4.0)
    phi = torch.tanh(2.0 * _smooth(gen, nx, ny, cells) + 0.02)
    s, _ = _strain(c["n0"], c["gdot"], c["dt"], nx, ny)
    qx, ky, k2, keep = _wavenumbers(nx, ny, c["dx"], s, "cuda")
    psi = torch.fft.rfft2(_smooth(gen, nx, ny, 2.0 * cells)) * keep
    speed = torch.fft.irfft2(1j * qx * psi, s=(ny, nx)).std()
    psi = psi * (0.1 * math.sqrt(8.0 / 9.0 * c["kappa"]) / c["eta"] / speed)
    omega = torch.fft.irfft2(k2 * psi, s=(ny, nx))
    psi = torch.fft.irfft2(psi, s=(ny, nx))
    if c["rho"] == 0.0:
        omega = torch.zeros_like(omega)
    return phi.to(dt), psi.to(dt), omega.to(dt)


def _params(c):
    return {k: c[k] for k in ("a", "b", "kappa", "M", "eta", "rho", "gdot", "dt")}


def _members(c):
    """The runs of an ensemble as step cases: sizes doubling from `small`, every
    second one without inertia, shear rates spread over 1e-4 .. 3e-2."""
    out = []
    for r in range(c["runs"]):
        n = c["small"] << (r * c["sizes"] // c["runs"])
        out.append(_step("", n, n, 32, c["steps"], c["n0"], rho=float(r % 2),
                         gdot=1e-4 * 300.0 ** (r / max(c["runs"] - 1, 1))))
    return out


_streams = []


def _stream():
    """The stream that this program's grids run on, one after the other: a run
    is timed by its own steps and not by what others overlap with it."""
    if not _streams:
        _streams.append(torch.cuda.Stream())
    return _streams[0]


def prepare(case, seed):
    c = case
    if c["kind"] == "ensemble":
        ms = _members(c)
        ens = shf.Ensemble([m["nx"] for m in ms], [m["ny"] for m in ms],
                           [[m[k] for k in ("a", "b", "kappa", "M", "eta", "rho", "gdot", "dt")] for m in ms],
                           precision=shf.SHF_FP32, stream=_stream())
        for r, m in enumerate(ms):
            ens.members[r].set_fields(*[f.double().cpu().numpy() for f in _fields(m, 1000 * seed + r)])
        ens.set_step(c["n0"])
        return dict(case=c, ens=ens)
    fields = _fields(c, seed)
    g = shf.Grid(c["nx"], c["ny"], c["dx"], shf.SHF_FP64 if c["prec"] == 64 else shf.SHF_FP32, stream=_stream())
    g.set_params(**_params(c))
    if c["kind"] == "host":
        src = [torch.empty(f.shape, dtype=f.dtype, pin_memory=True) for f in fields]
        out = [torch.empty(f.shape, dtype=f.dtype, pin_memory=True) for f in fields]
        for d, f in zip(src, fields):
            d.copy_(f)
        torch.cuda.synchronize()
        g.set_step(c["n0"])
        return dict(case=c, grid=g, keep=(src, out), src=[t.numpy() for t in src], out=[t.numpy() for t in out])
    state = [torch.empty_like(f) for f in fields]
    g.bind_device_fields(*state)
    for d, f in zip(state, fields):
        d.copy_(f)
    torch.cuda.synchronize()
    g.set_step(c["n0"])
    return dict(case=c, grid=g, fields=state[:2] if c["rho"] == 0.0 else state)


def run(state):
    c = state["case"]
    if c["kind"] == "ensemble":
        ens = state["ens"]
        ens.step(c["steps"])
        out = []
        for r, m in enumerate(ens.members):
            f = shf.shf_get_fields_f32(m.handle, m.nx, m.ny)
            out.append(f if r % 2 else f[:2])
        return out
    g = state["grid"]
    if c["kind"] == "step":
        g.step(c["steps"])
        return state["fields"]
    if c["kind"] == "host":
        return list(g.step_host_f32(c["steps"], *state["src"], out=state["out"]))[:2 if c["rho"] == 0.0 else 3]
    moments, bins = g.structure_factor(c["bins"])
    G, lengths = g.gradient_tensor()
    return dict(moments=moments, bins=bins, tensor=np.array(G), lengths=np.array(lengths), mass=g.mass())


def work(case):
    """Bytes: the state in and out once; operations: the real 2D transforms at
    2.5 log2(N) per point and the stencils and multipliers."""
    c = case
    if c["kind"] == "ensemble":
        ws = [work(m) for m in _members(c)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    n, real = c["nx"] * c["ny"], c["prec"] // 8
    if c["kind"] == "observables":
        return {"bytes": n * real, "flops": n * (2.5 * math.log2(n) + 15)}
    stokes = c["rho"] == 0.0
    transforms, fields, point = (5, 2, 80) if stokes else (7, 3, 110)
    return {"bytes": 2 * fields * n * real, "flops": c["steps"] * n * (transforms * 2.5 * math.log2(n) + point)}


# ---------------------------------------------- the same in plain torch, 64 bits

def _at(f, di, dj):
    return torch.roll(f, (-dj, -di), dims=(0, 1))


def _dx(f, h):
    return (_at(f, 1, 0) - _at(f, -1, 0)) / (2.0 * h)


def _dy(f, s, h):
    d = -2 if s >= 0.0 else 2
    w = 0.5 * abs(s)
    return ((1.0 - w) * (_at(f, 0, 1) - _at(f, 0, -1)) + w * (_at(f, d, 1) - _at(f, -d, -1))) / (2.0 * h)


def _bracket(p, f, s, h):
    """J(p, f) = d_y p d_x f - d_x p d_y f, sheared."""
    return _dy(p, s, h) * _dx(f, h) - _dx(p, h) * _dy(f, s, h)


def _relabel(f, cells):
    """Row j moved by j * cells points along x."""
    ny, nx = f.shape
    j = torch.arange(ny, device=f.device)[:, None]
    i = torch.arange(nx, device=f.device)[None, :]
    return torch.gather(f, 1, (i - j * cells) % nx)


def _exact_steps(c, phi, psi, om):
    nx, ny, h, dt, rho = c["nx"], c["ny"], c["dx"], c["dt"], c["rho"]
    r = nx // ny
    back = lambda z: torch.fft.irfft2(z, s=(ny, nx))  # noqa: E731
    for n in range(c["n0"], c["n0"] + c["steps"]):
        s0, K0 = _strain(n, c["gdot"], dt, nx, ny)
        s1, K1 = _strain(n + 1, c["gdot"], dt, nx, ny)
        # advection, then the diffusive update of phi at s^n
        star = phi - dt * _bracket(psi, phi, s0, h)
        if rho > 0.0:
            om = om - dt * _bracket(psi, om, s0, h)
        qx, ky, k2, keep = _wavenumbers(nx, ny, h, s0, phi.device)
        c4 = 0.5 * dt * c["kappa"] * c["M"] * k2 * k2
        P = torch.fft.rfft2(star)
        Q = torch.fft.rfft2(phi * phi * phi)
        phi = back(((1.0 - c4 + dt * c["a"] * c["M"] * k2) * P - dt * c["b"] * c["M"] * k2 * Q) / (1.0 + c4) * keep)
        if K1 != K0:
            phi = _relabel(phi, (K1 - K0) * r)
            om = _relabel(om, (K1 - K0) * r)
        # the force and the flow at s^{n+1}
        lap = ((1.0 + s1 * s1) * (_at(phi, 1, 0) - 2.0 * phi + _at(phi, -1, 0)) / (h * h)
               - 2.0 * s1 * (_at(phi, 1, 1) - _at(phi, 1, -1) - _at(phi, -1, 1) + _at(phi, -1, -1)) / (4.0 * h * h)
               + (_at(phi, 0, 1) - 2.0 * phi + _at(phi, 0, -1)) / (h * h))
        mu = phi * (c["b"] * phi * phi - c["a"]) - c["kappa"] * lap
        G = torch.fft.rfft2(-_bracket(mu, phi, s1, h))  # minus the force's curl
        qx, ky, k2, keep = _wavenumbers(nx, ny, h, s1, phi.device)
        keep[0, 0] = 0.0
        k2[0, 0] = 1.0
        if rho > 0.0:
            cc = 0.5 * dt * (c["eta"] / rho) * k2
            W = ((1.0 - cc) * torch.fft.rfft2(om) + dt / rho * G) / (1.0 + cc) * keep
            om, psi = back(W), back(W / k2)
        else:
            psi = back(G / (c["eta"] * k2 * k2) * keep)
    return (phi, psi) if rho == 0.0 else (phi, psi, om)


def _exact_observables(c, phi):
    nx, ny, h = c["nx"], c["ny"], c["dx"]
    s, _ = _strain(c["n0"], c["gdot"], c["dt"], nx, ny)
    qx, ky, k2, keep = _wavenumbers(nx, ny, h, s, phi.device)
    S = torch.fft.rfft2(phi).abs().square() / float(nx * ny) ** 2 * keep
    S[:, 1:] *= 2.0
    den = S.sum()
    qx = qx.expand_as(ky)
    G = [float((u * v * S).sum() / den) for u, v in ((qx, qx), (qx, ky), (ky, ky))]
    mid, rad = 0.5 * (G[0] + G[2]), math.hypot(0.5 * (G[0] - G[2]), G[1])
    ell = math.sqrt(c["kappa"] / c["a"])
    k2[0, 0] = 1.0
    S[0, 0] = 0.0
    k = k2.sqrt()
    m = [float(S.sum()), float((k * S).sum()), float((S / k).sum())]
    m += [2.0 * math.pi * m[0] / m[1], m[2] / m[0]]
    return dict(moments=np.array(m), bins=None, tensor=np.array(G),
                lengths=np.array([1.0 / (ell * (mid - rad)), 1.0 / (ell * (mid + rad))]), mass=float(phi.mean()))


def exact(case, seed):
    """The outputs of run() in float64 (the bins are left out: a mode that lies
    on the edge of a bin may fall on either side of it)."""
    c = case
    if c["kind"] == "ensemble":
        return [_exact_steps(m, *[f.double() for f in _fields(m, 1000 * seed + r)])
                for r, m in enumerate(_members(c))]
    fields = [f.double() for f in _fields(c, seed)]
    if c["kind"] == "observables":
        return _exact_observables(c, fields[0])
    return list(_exact_steps(c, *fields))
