"""The radial bins of the structure factor at the edges of its kernel's range
(fewer threads than a warp, one column per CTA, long and flat boxes, strains
of either sign) against a plain float64 transform.  A mode whose k lies within
rounding of a bin's edge may fall on either side, so the running sums of the
bins are held between the sums of the modes surely and possibly below each
edge; the tolerances are the transform's rounding (eps log2 N of the total)."""
import math

import numpy as np
import pytest

import paper_0710_5912_gb300 as shf
from paper_0710_5912_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,eps", [(shf.SHF_FP64, 2.3e-16), (shf.SHF_FP32, 1.2e-7)])
@pytest.mark.parametrize("nbins", [1, 7, 3000])
@pytest.mark.parametrize("shape,dx,strain", [((16, 16), 1.0, 0.0), ((32, 16), 0.9, -0.4), ((64, 64), 1.0, 0.5 - 2 ** -10),
                                             ((256, 64), 0.37, 1.7), ((128, 128), 2.0, 0.0), ((1024, 512), 1 / 512, -0.9),
                                             ((4096, 16), 1.0, 3.0)])
def test_bins_hold_the_modes_below_each_edge(prec, eps, nbins, shape, dx, strain):
    nx, ny = shape
    phi = inputs.quench_noise(nx, ny, 5, 0.5) + 0.1
    if prec == shf.SHF_FP32:
        phi = phi.astype(np.float32).astype(np.float64)
    with shf.Grid(nx, ny, dx, prec) as g:
        g.set_params(gdot=strain, dt=1.0)
        g.set_fields(phi)
        g.set_step(1)                                   # s = gdot dt, no wrap at these strains
        s = g.get_time()[2]
        moments, bins = g.structure_factor(nbins)
    assert s == strain
    S = np.abs(np.fft.fft2(phi)) ** 2 / float(nx * ny) ** 2
    m = np.fft.fftfreq(nx, 1.0 / nx)[None, :]
    n = np.fft.fftfreq(ny, 1.0 / ny)[:, None]
    keep = (np.abs(m) < nx // 2) & (n != -(ny // 2)) & ((m != 0) | (n != 0))
    qx = 2 * math.pi / (nx * dx) * m
    k = np.hypot(qx, 2 * math.pi / (ny * dx) * n - s * qx) / (2 * math.pi / (ny * dx))
    S, k = S[keep], k[keep]
    tol = 4 * eps * math.log2(nx * ny) * (S.sum() + 0.01)
    run = np.cumsum(bins.astype(np.longdouble))         # (500,000 additions in float64 would cost more than tol)
    order = np.argsort(k)
    total = np.concatenate([[np.longdouble(0)], np.cumsum(S[order].astype(np.longdouble))])
    edge = np.arange(1, nbins + 1, dtype=np.float64)
    below = total[np.searchsorted(k[order], edge * (1 - 1e-12))]
    upto = total[np.searchsorted(k[order], edge * (1 + 1e-12))]
    assert np.all(run >= below - tol) and np.all(run <= upto + tol)
    assert abs(moments[0] - float(total[-1])) <= tol
