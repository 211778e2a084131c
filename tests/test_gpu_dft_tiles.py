"""The temporal DFT at the edges of its tile rule (csrc/iter_kernels.cu: 32 pixels up to 128 an SM and from
five frames on, else 64), and over the lengths of a single stage.  Bar: the solver's 1e-5."""

import numpy as np
import pytest

import oracle
from test_gpu_fft_lengths import gpu, problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Nx,Ny,Nt", [(152, 128, 5), (153, 128, 5), (152, 128, 4)] + [(21, 20, t) for t in (1, 2, 3, 4, 5, 6, 7, 8)])
def test_solve(Nx, Ny, Nt):
    from paper_1203_4587_gb300 import Plan
    c = problem(Nx, Ny, Nt, 2)
    P = Plan(c.mask.astype(np.uint8), gpu(c.sens), 0.01, c.mu, prior="dft", max_iters=3)
    x, info = P.solve(gpu(c.kspace))
    xr, oi = oracle.Problem(c.kspace, c.sens, c.mask, c.mu).solve("dft", 0.01, c.mu, c.rho, 3)
    assert np.linalg.norm(x.cpu().numpy() - xr) <= 1e-5 * np.linalg.norm(xr)
    assert abs(info.J - oi["J"][-1]) <= 1e-5 * oi["J"][-1]
