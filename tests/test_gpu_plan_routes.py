"""Which inversion a plan takes: the tensor-core form (csrc/plan_tc.cu) or the double-float sweep
(csrc/plan_kernels.cu), and that the rule holds what each form promises."""

import numpy as np
import pytest

import oracle
import synthdata

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def inverses(sens, mask, mu, cols, **opts):
    from paper_1203_4587_gb300 import Plan
    P = Plan(mask.astype(np.uint8), torch.from_numpy(sens).cuda(), 0.01, mu, max_iters=1, **opts)
    out = torch.stack([P.export_inverse(i, t) for i in range(cols) for t in range(mask.shape[0])])
    P.close()
    return torch.view_as_real(out)


@pytest.mark.parametrize("storage", ["fp16", "bf16"])
def test_16_bit_inverses_are_the_sweeps(storage):
    """A further image column of ten times the sensitivity lifts the condition bound above the
    tensor-core form's, so its plan is inverted by the sweep: the common columns' 16-bit inverses are the
    same bits, also where a value lies next to a rounding tie."""
    sens = synthdata.make_sens(65, 256, 12, phase_y=0.3).astype(np.complex64)
    sens[:, :, 64] *= 10
    mask = synthdata.make_mask(256, 8, 6, np.random.default_rng(1))
    a = inverses(np.ascontiguousarray(sens[:, :, :64]), mask, 0.02, 64, storage=storage)   # bound 51
    assert torch.equal(a, inverses(sens, mask, 0.02, 64, storage=storage))


# coils of 1e-18 and 1e18: products and their low halves reach the ends of the FP32 range
@pytest.mark.parametrize("scale,mu", [(1e-18, 1e-37), (1e-9, 1e-18), (1e9, 1e17), (1e18, 1e35)])
def test_blocks_far_from_one_in_scale(scale, mu):
    """Half an FP32 ulp (a subnormal's at the least) plus 2^-41 max|A|, the bar at usual scales."""
    from paper_1203_4587_gb300 import binding
    sens = (scale * synthdata.make_sens(2, 72, 3, phase_y=0.3)).astype(np.complex64)
    mask = synthdata.make_mask(72, 1, 3, np.random.default_rng(2))
    cols = torch.from_numpy(np.ascontiguousarray(sens.transpose(2, 0, 1))).cuda()
    A = binding.gram_inverse_noalloc(torch.from_numpy(np.repeat(mask, 2, axis=0).astype(np.uint8)).cuda(), cols, mu).cpu().numpy()
    ref = oracle.inverse_blocks(oracle.gram_blocks(sens.astype(np.complex128), mask, [1])[0, 0], float(np.float32(mu)))
    top = np.abs(ref).max()
    for part in (np.real, np.imag):
        a, r = part(A[1]).astype(np.float64), part(ref)
        half = np.maximum(2.0 ** (np.floor(np.log2(np.maximum(np.abs(r), 1e-300))) - 24), 2.0 ** -150)
        assert np.all(np.abs(a - r) <= half + 2.0 ** -41 * top)


def launches(call):
    from paper_1203_4587_gb300 import binding
    n = binding.kernel_launches()
    call()
    return binding.kernel_launches() - n


# on 152 SMs: 96 and above always, 80 with 16 blocks, 64 with two blocks an SM, 56 with four, never below;
# 416 is the largest size (csrc/host_logic.h)
@pytest.mark.parametrize("Ny,Nx,Nt,tensor", [(48, 160, 8, False), (55, 160, 8, False), (56, 75, 8, False), (56, 76, 8, True),
                                             (64, 37, 8, False), (64, 38, 8, True), (80, 3, 5, False), (80, 2, 8, True),
                                             (96, 1, 1, True), (416, 1, 1, True), (417, 1, 1, False)])
def test_plan_route_by_size(Ny, Nx, Nt, tensor):
    """Small plans are not slower for the tensor cores' launches: the sweep is two kernels (three with the
    condition's bound), the tensor-core form five a chunk and three more."""
    from paper_1203_4587_gb300 import Plan
    sens = synthdata.make_sens(Nx, Ny, 2, phase_y=0.3).astype(np.complex64)
    mask = synthdata.make_mask(Ny, Nt, 3, np.random.default_rng(Ny))
    P = Plan(mask.astype(np.uint8), torch.from_numpy(sens).cuda(), 0.01, 0.1, max_iters=1)
    n = launches(lambda: P.set_mu(0.1))
    assert n >= 8 if tensor else n <= 3
    P.close()


# a chunk of 16 MiB holds 72 blocks up to 64, 32 up to 96
@pytest.mark.parametrize("Ny,nblk,tensor", [(32, 1, False), (33, 60, True), (33, 130, False), (36, 130, True), (40, 256, False),
                                            (44, 200, True), (44, 512, False), (48, 1024, True), (65, 256, True),
                                            (65, 1024, False), (72, 1024, True)])
def test_blocks_route_by_size(Ny, nblk, tensor):
    from paper_1203_4587_gb300 import binding
    sens = torch.full((nblk, 2, Ny), 0.7, dtype=torch.complex64, device="cuda")
    mask = (torch.arange(Ny, device="cuda") % 3 == 0).to(torch.uint8).repeat(nblk, 1)
    n = launches(lambda: binding.gram_inverse_noalloc(mask, sens, 0.1))
    assert n >= 8 if tensor else n <= 3


@pytest.mark.parametrize("Ny", [56, 63, 64, 65, 72, 80, 95])
def test_small_sizes_on_the_tensor_cores(Ny):
    """Enough blocks for the tensor-core form below 96: tile edges and padding, as test_gpu_plan_tc.py."""
    from test_gpu_plan_tc import check
    check(Ny, 0.1, Nx=77, Nt=8)


def test_ill_conditioned_and_non_finite_blocks_of_the_tensor_cores_sizes():
    """Two kernels for the bounds and the FP64 one; a well-conditioned call afterwards takes the six of the
    tensor cores."""
    from paper_1203_4587_gb300 import binding
    lib = binding.load()
    Ny = 40
    sens = synthdata.make_sens(3, Ny, 3, phase_y=0.3).astype(np.complex64)
    mask = synthdata.make_mask(Ny, 1, 3, np.random.default_rng(4))
    m = torch.from_numpy(np.repeat(mask, 3, axis=0).astype(np.uint8)).cuda()
    cols = torch.from_numpy(np.ascontiguousarray(sens.transpose(2, 0, 1))).cuda()
    for mu in (0.005, 0.1):
        A = binding.gram_inverse_noalloc(m, cols, mu).cpu().numpy()
        assert launches(lambda: binding.gram_inverse_noalloc(m, cols, mu)) == (3 if mu < 0.01 else 8)
        ref = oracle.inverse_blocks(oracle.gram_blocks(sens.astype(np.complex128), mask, [2])[0, 0], float(np.float32(mu)))
        top = np.abs(ref).max()
        for part in (np.real, np.imag):
            a, r = part(A[2]).astype(np.float64), part(ref)
            assert np.all(np.abs(a - r) <= 0.5 * np.spacing(np.abs(r).astype(np.float32)) + 2.0 ** -41 * top)
    bad = cols.clone()
    bad[1, 0, 3] = complex(float("inf"), 0.0)
    out = torch.empty((3, Ny, Ny), dtype=torch.complex64, device="cuda")
    assert lib.recon_gram_inverse_noalloc(Ny, 3, 3, binding._ptr(m), binding._ptr(bad), 0.1, binding._ptr(out), None) == 6
