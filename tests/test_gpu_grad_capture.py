"""The reverse pass keeps its last segment's inner states from the forward only while nothing else can
have written them: segment lengths that leave several segments, a second backward, and graphs of the
forward and the backward replayed between direct calls.

The launches of a pair of calls are the same with and without captures around them, so dL/dy has the same
bits as from an engine of its own."""

import ctypes as C

import numpy as np
import pytest

from test_gpu_grad import gpu, host, make, plan_for

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

K = 7


def ptrs(t):
    return (C.c_void_p * 1)(t.data_ptr())


@pytest.fixture(scope="module")
def case():
    return make("tiny", Nx=19, Ny=27, Nt=5, Nc=3)


def own(case, y, xb, every):
    from paper_1203_4587_gb300 import Grad
    G = Grad([plan_for(case, K)], checkpoint_every=every)
    G.forward([y])
    return host(G.backward([xb])[0][0])


@pytest.mark.parametrize("every", [2, 3, 5])
def test_second_backward(case, every):
    from paper_1203_4587_gb300 import Grad
    y, xb = gpu(case.kspace), gpu(case.x_true)
    ref = own(case, y, xb, every)
    G = Grad([plan_for(case, K)], checkpoint_every=every)
    G.forward([y])
    for _ in range(3):
        assert np.array_equal(host(G.backward([xb])[0][0]), ref)


@pytest.mark.parametrize("every", [2, 3, 5])
def test_replays_between_direct_calls(case, every):
    """A replayed backward leaves the first segment where a direct forward had left the last one; a
    replayed forward leaves another input's."""
    from paper_1203_4587_gb300 import Grad, binding
    lib = binding.load()
    y1, xb = gpu(case.kspace), gpu(case.x_true)
    y2 = gpu(2j * case.kspace[::-1].copy())
    ref1, ref2 = own(case, y1, xb, every), own(case, y2, xb, every)
    G = Grad([plan_for(case, K)], checkpoint_every=every)
    G.forward([y1])
    G.backward([xb])
    y, img, gy = y1.clone(), torch.empty_like(xb), torch.empty_like(y1)
    fwd, bwd = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(fwd):
        s = C.c_void_p(torch.cuda.current_stream().cuda_stream)
        assert lib.recon_grad_forward(G._h, ptrs(y), ptrs(img), s) == 0
    with torch.cuda.graph(bwd):
        s = C.c_void_p(torch.cuda.current_stream().cuda_stream)
        assert lib.recon_grad_backward(G._h, ptrs(xb), ptrs(gy), None, None, s) == 0
    G.forward([y1])
    bwd.replay()
    torch.cuda.synchronize()
    assert np.array_equal(host(gy), ref1)
    assert np.array_equal(host(G.backward([xb])[0][0]), ref1)
    y.copy_(y2)
    G.forward([y1])
    fwd.replay()
    torch.cuda.synchronize()
    assert np.array_equal(host(G.backward([xb])[0][0]), ref2)
    fwd.replay()
    bwd.replay()
    torch.cuda.synchronize()
    assert np.array_equal(host(gy), ref2)
