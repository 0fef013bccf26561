"""Steps recorded into a caller's CUDA graph: an unreplayed capture leaves the
grid as it was, and a replay forms the strain of the counter it finds."""
import numpy as np
import pytest

import paper_0710_5912_gb300 as shf
from paper_0710_5912_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PARAMS = dict(a=1.0, b=1.0, kappa=1.0, M=1.0, eta=0.7, gdot=0.4, dt=0.01)


def start(g, rho, n0):
    nx, ny = g.nx, g.ny
    g.set_fields(inputs.quench_noise(nx, ny, 3, 0.5), inputs.quench_noise(nx, ny, 4, 0.05),
                 inputs.quench_noise(nx, ny, 5, 0.05) * (rho > 0))
    g.set_step(n0)


@pytest.mark.parametrize("prec,rho", [(shf.SHF_FP64, 0.8), (shf.SHF_FP64, 0.0), (shf.SHF_FP32, 0.0)])
def test_captured_steps(prec, rho):
    stream = torch.cuda.Stream()
    with shf.Grid(64, 32, 1.0, prec) as ref, shf.Grid(64, 32, 1.0, prec, stream=stream) as g:
        for grid in (ref, g):
            grid.set_params(rho=rho, **PARAMS)
        start(ref, rho, 249)                            # the strain wraps in this step
        ref.step(1)
        want = ref.get_fields()
        start(g, rho, 10)
        g.step(2)                                       # its state is kept from here on
        g.sync()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            g.step(1)
        start(g, rho, 249)
        with torch.cuda.stream(stream):
            graph.replay()
        for a, b in zip(g.get_fields(), want):
            assert np.array_equal(a, b)
        start(g, rho, 249)
        with torch.cuda.graph(torch.cuda.CUDAGraph(), stream=stream):
            g.step(1)                                   # never replayed
        g.step(1)
        for a, b in zip(g.get_fields(), want):
            assert np.array_equal(a, b)
