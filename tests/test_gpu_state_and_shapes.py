"""The step state kept between calls follows new parameters, and small grids give
the same bits in the launch shapes that only a full chip takes.

New gdot and dt (no shf_set_step) change the strain of the very next step, here
into one that wraps.  Small grids: as one of so many members that thread groups
and single instances per CTA are given up, the same bits as alone.  Tolerances
are those of the single-step parity tests."""
import numpy as np
import pytest

import oracle
import paper_0710_5912_gb300 as shf
from paper_0710_5912_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FP32, FP64 = shf.SHF_FP32, shf.SHF_FP64
TOL = {FP64: 1e-11, FP32: 1e-5}
NAMES = ("phi", "psi", "omega")


def row(p):
    return [p.a, p.b, p.kappa, p.M, p.eta, p.rho, p.gdot, p.dt]


def state(nx, ny, rho, amp=0.5):
    return (inputs.quench_noise(nx, ny, 27, amp), inputs.quench_noise(nx, ny, 28, 0.05),
            inputs.quench_noise(nx, ny, 29, 0.05) * (rho > 0))


def close(got, want, tol, rho):
    for name, a, b in zip(NAMES, got, want):
        if name == "omega" and rho == 0:
            assert not a.any()
        else:
            err = np.linalg.norm(a - b) / np.linalg.norm(b)
            assert err <= tol, f"{name}: {err:.2e}"


@pytest.mark.parametrize("prec", [FP64, FP32])
@pytest.mark.parametrize("rho", [0.0, 0.7])
def test_new_shear_rate_and_time_step_reach_the_next_step(prec, rho):
    nx, ny, n = 64, 32, 30
    p1 = oracle.Params(a=0.9, b=1.1, kappa=0.8, M=1.2, eta=0.6, rho=rho, gdot=0.3, dt=0.005, dx=0.9)
    p2 = oracle.Params(a=0.9, b=1.1, kappa=0.8, M=1.2, eta=0.6, rho=rho, gdot=-6.2, dt=0.01 * 17 / 33, dx=0.9)
    K = [oracle.strain(n + i, p2.gdot, p2.dt, nx, ny)[1] for i in range(3)]
    assert len(set(K)) == 2                             # a wrap on the way, under the new parameters only
    assert len({oracle.strain(n - 3 + i, p1.gdot, p1.dt, nx, ny)[1] for i in range(6)}) == 1
    first = state(nx, ny, rho)
    with shf.Grid(nx, ny, p1.dx, prec) as g, shf.Grid(nx, ny, p1.dx, prec) as fresh:
        g.set_params(*row(p1))
        g.set_fields(*first)
        g.set_step(n - 3)
        g.step(3)
        mid = g.get_fields()
        g.set_params(*row(p2))
        g.step(2)
        got = g.get_fields()
        fresh.set_params(*row(p2))
        fresh.set_fields(*mid)
        fresh.set_step(n)
        fresh.step(2)
        for name, a, b in zip(NAMES, got, fresh.get_fields()):
            assert np.array_equal(a, b), name
    close(got, oracle.run(*mid, 2, p2, n0=n), TOL[prec], rho)
    ens = shf.Ensemble([nx] * 3, [ny] * 3, [row(p1)] * 3, dx=[p1.dx] * 3, precision=prec)
    for m in ens.members:
        m.set_fields(*first)
    ens.set_step(n - 3)
    ens.step(3)
    shf.shf_set_params(ens.members[1].handle, *row(p2))
    ens.step(2)
    for name, a, b in zip(NAMES, ens.members[1].get_fields(), got):
        assert np.array_equal(a, b), f"member {name}"
    close(ens.members[0].get_fields(), oracle.run(*first, 5, p1, n0=n - 3), TOL[prec], rho)
    ens.close()


@pytest.mark.parametrize("prec", [FP64, FP32])
@pytest.mark.parametrize("rho", [0.0, 0.7])
@pytest.mark.parametrize("shape", [(32, 32), (64, 16)])
def test_small_members_of_a_full_chip_match_a_grid_alone(prec, rho, shape):
    nx, ny = shape
    p = oracle.Params(a=0.9, b=1.1, kappa=0.8, M=1.2, eta=0.6, rho=rho, gdot=0.3, dt=0.01, dx=0.9)
    fields = state(nx, ny, rho, 0.5 * ny / nx)
    points = 8 if prec == FP64 else 16
    nm = 1 + 160 * 768 // (2 * (nx // points) * (ny // 2))   # two groups of every row pair no longer fit 152 SMs
    ens = shf.Ensemble([nx] * nm, [ny] * nm, [row(p)] * nm, dx=[p.dx] * nm, precision=prec)
    ens.members[nm - 1].set_fields(*fields)
    with shf.Grid(nx, ny, p.dx, prec) as g:
        g.set_params(*row(p))
        g.set_fields(*fields)
        for x in (g, ens):
            x.set_step(37)
            x.step(2)
        for name, a, b in zip(NAMES, g.get_fields(), ens.members[nm - 1].get_fields()):
            assert np.array_equal(a, b), name
    ens.close()
