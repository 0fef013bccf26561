"""The launch shapes of the step's kernels (thread groups per item, instances
per CTA, the grouped column kernel) at the edges of their ranges: the smallest
rows and columns, long rows with few of them, sizes on either side of the
lines.  A launch's shape depends on how much work it has, so a single grid and
a member of a large ensemble of the same size take different ones: both give
the same bits, and inertial runs agree with the oracle at the tolerances of
the single-step parity tests.  The strain wraps on the way."""
import numpy as np
import pytest

import oracle
import paper_0710_5912_gb300 as shf
from paper_0710_5912_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FP32, FP64 = shf.SHF_FP32, shf.SHF_FP64
TOL = {FP64: 1e-11, FP32: 1e-5}
SHAPES = [(32, 32), (64, 16), (128, 128), (256, 64), (512, 512), (1024, 16), (1024, 256), (2048, 32), (2048, 512),
          (4096, 64)]


@pytest.mark.parametrize("prec", [FP64, FP32])
@pytest.mark.parametrize("rho", [0.0, 0.7])
@pytest.mark.parametrize("shape", SHAPES)
def test_launch_shapes_give_the_same_bits_and_match_oracle(prec, rho, shape):
    nx, ny = shape
    r = nx // ny
    p = oracle.Params(a=0.9, b=1.1, kappa=0.8, M=1.2, eta=0.6, rho=rho, gdot=0.3, dt=0.01, dx=0.9)
    n0 = int(np.ceil(0.5 * r / (p.gdot * p.dt))) - 1     # the strain passes r / 2 in the first step
    assert oracle.strain(n0, p.gdot, p.dt, nx, ny)[1] != oracle.strain(n0 + 1, p.gdot, p.dt, nx, ny)[1]
    fields = (inputs.quench_noise(nx, ny, 17, 0.5 / r), inputs.quench_noise(nx, ny, 18, 0.05),
              inputs.quench_noise(nx, ny, 19, 0.05) * (rho > 0))
    row = [p.a, p.b, p.kappa, p.M, p.eta, p.rho, p.gdot, p.dt]
    with shf.Grid(nx, ny, p.dx, prec) as g:
        g.set_params(*row)
        g.set_fields(*fields)
        g.set_step(n0)
        g.step(2)
        g.sync()
        got = g.get_fields()
    # enough members that all of a launch's items no longer fit on the chip at once
    nm = min(100, 2 + (152 * 768 * 2) // max(1, (nx // 16) * (ny // 2)))
    ens = shf.Ensemble([nx] * nm, [ny] * nm, [row] * nm, dx=[p.dx] * nm, precision=prec)
    ens.members[nm - 1].set_fields(*fields)
    ens.set_step(n0)
    ens.step(2)
    ens.sync()
    for name, a, b in zip(("phi", "psi", "omega"), got, ens.members[nm - 1].get_fields()):
        assert np.array_equal(a, b), f"{shape} {name}"
    ens.close()
    if rho > 0:
        want = oracle.run(*fields, 2, p, n0=n0)
        for name, a, b in zip(("phi", "psi", "omega"), got, want):
            err = np.linalg.norm(a - b) / np.linalg.norm(b)
            assert err <= TOL[prec], f"{shape} {name}: {err:.2e}"
