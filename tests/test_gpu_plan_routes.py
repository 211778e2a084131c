"""Which inversion a plan takes: the tensor-core form (csrc/plan_tc.cu) or the double-float sweep
(csrc/plan_kernels.cu), and that the rule holds what each form promises."""

import numpy as np
import pytest

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
