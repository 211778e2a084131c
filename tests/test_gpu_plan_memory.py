"""recon_plan_set_mu (and with it plan creation) when device memory is short: the tensor-core inversion
takes smaller chunks, then the double-float sweep takes its place, and the inverses are the same."""

import gc

import numpy as np
import pytest

import synthdata

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MB = 1 << 20


def fill_to(free_mb):
    """Tensors that leave about free_mb of the device."""
    held = []
    for _ in range(4):
        torch.cuda.synchronize()
        rest = torch.cuda.mem_get_info()[0] - free_mb * MB
        if rest < 2 * MB:
            break
        held.append(torch.empty(rest // (2 * MB) * (2 * MB), dtype=torch.uint8, device="cuda"))
    return held


def plan(Nx, Ny, Nt, scale=1.0):
    from paper_1203_4587_gb300 import Plan
    sens = (scale * synthdata.make_sens(Nx, Ny, 3, phase_y=0.3)).astype(np.complex64)
    mask = synthdata.make_mask(Ny, Nt, 3, np.random.default_rng(Ny))
    return Plan(mask.astype(np.uint8), torch.from_numpy(sens).cuda(), 0.01, 0.1, max_iters=1)


def launches(P):
    from paper_1203_4587_gb300 import binding
    n = binding.kernel_launches()
    P.set_mu(0.1)
    return binding.kernel_launches() - n


def ends(P, Nx, Nt):
    return torch.stack([P.export_inverse(i, t) for i in (0, Nx // 2, Nx - 1) for t in (0, Nt - 1)])


# 64 columns of 16 frames, 128 x 128: chunks of 38 columns (558 MB) as they come, 8 or 9 in 150 MB
@pytest.mark.parametrize("Nx,Ny,Nt,free_mb,chunks", [(64, 128, 16, 150, True), (8, 64, 128, 24, False)])
def test_set_mu_with_little_memory(Nx, Ny, Nt, free_mb, chunks):
    """(8 columns of 128 frames of 64 x 64: one column takes 38 MB, the sweep 10 MB.)"""
    sweep = plan(2, Ny, 2, scale=10.0)   # condition bound above 64: the sweep's launches, its code loaded
    few = launches(sweep)
    P = plan(Nx, Ny, Nt)
    usual = launches(P)
    before = ends(P, Nx, Nt)
    assert usual > few
    gc.collect()
    torch.cuda.empty_cache()
    held = fill_to(free_mb)
    n = launches(P)
    del held
    torch.cuda.empty_cache()
    assert n > usual if chunks else n <= few + 1   # + 1: the coils' power
    after = ends(P, Nx, Nt)
    if chunks:
        assert torch.equal(torch.view_as_real(after), torch.view_as_real(before))
    else:   # one rounding of results good to 2^-43
        assert float((after - before).abs().max()) <= 2.0 ** -23 * float(before.abs().max())
