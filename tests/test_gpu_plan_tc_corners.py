"""The tensor-core inversion (csrc/plan_tc.cu) where it keeps the fewest digits: condition bounds just
under its limit of 64, the largest sizes, few and many sampled rows, and structured operands (one coil of
constant magnitude: C_t alone decides M).

Bar: every element within half an FP32 ulp of the 64-bit inverse plus 2^-41 max|A|.  What adds up to less:
E^2 from 11-bit operands 2^-43, M's rounding in double-float 2^-48 times the condition 2^-43, E's integers
2^-45, the 64-bit reference 2^-45."""

import numpy as np
import pytest

import oracle
import synthdata

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NX = 2


def coils(kind, Ny):
    if kind == "coils":
        return synthdata.make_sens(NX, Ny, 4, phase_y=0.3).astype(np.complex64)
    j = np.arange(Ny) / Ny
    phase = np.exp(3.4j * j) if kind == "phase" else np.ones(Ny)
    return np.repeat(phase[None, :, None], NX, axis=2).astype(np.complex64)


def rows(kind, Ny):
    rng = np.random.default_rng(Ny)
    m = np.zeros((1, Ny), bool)
    m[0, rng.choice(Ny, Ny // (2 if kind == "half" else 10), replace=False)] = True
    m[0, :4] = True
    return m


def excess(A, ref):
    """The largest distance from ref beyond half an FP32 ulp, over max|ref|."""
    worst = 0.0
    for part in (np.real, np.imag):
        a, r = part(A).astype(np.float64), part(ref)
        half = 2.0 ** (np.floor(np.log2(np.maximum(np.abs(r), 1e-300))) - 24)
        worst = max(worst, float(np.max(np.abs(a - r) - half)))
    return worst / np.abs(ref).max()


@pytest.mark.parametrize("cond", [63.0, 11.0])
@pytest.mark.parametrize("mask", ["half", "low"])
@pytest.mark.parametrize("kind", ["flat", "phase", "coils"])
@pytest.mark.parametrize("Ny", [96, 256, 384, 416])
def test_accuracy_at_the_corners(Ny, kind, mask, cond):
    from paper_1203_4587_gb300 import Plan
    sens, m = coils(kind, Ny), rows(mask, Ny)
    mu = float(np.float32((np.abs(sens.astype(np.complex128)) ** 2).sum(0).max() / (cond - 1)))
    P = Plan(m.astype(np.uint8), torch.from_numpy(sens).cuda(), 0.01, mu, max_iters=1)
    A = P.export_inverse(NX - 1, 0).cpu().numpy()
    P.close()
    ref = oracle.inverse_blocks(oracle.gram_blocks(sens.astype(np.complex128), m, [NX - 1])[0, 0], mu)
    assert excess(A, ref) <= 2.0 ** -41
