"""The closure's gradient in a CUDA graph that the caller captures (no host
loss, so nothing synchronises): captured with a closure that has trained on
nothing yet, on a smaller mesh and on the same one, and replayed after the
closure went on to larger meshes: the bits of a direct call."""
import ctypes

import numpy as np
import pytest

from paper_1408_5715_gb300 import binding as B
from paper_1408_5715_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _sample(nx, ny):
    mi = W.channel_bump(nx, ny, seed=2)
    m = B.Mesh.from_input(mi, "f32")
    m.upload()
    U = W.random_smooth_state(mi.centroids(), 1)
    return m, *(torch.tensor(x, dtype=torch.float32, device="cuda") for x in (U, 1.01 * U))


def _grad_without_loss(cl, sample, grad):
    m, U0, Ut = sample
    w = np.ones(4)
    B._check(B.load().fv_closure_loss_grad(
        m._h, ctypes.c_void_p(U0.data_ptr()), ctypes.c_void_p(Ut.data_ptr()), 1e-3,
        w.ctypes.data_as(ctypes.c_void_p), cl._h, None, ctypes.c_void_p(grad.data_ptr()),
        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))


@pytest.mark.parametrize("before", [None, (10, 6), (40, 20)])
def test_captured_gradient_outlives_larger_meshes(before):
    theta = (np.random.default_rng(0).normal(size=B.CLOSURE_PARAMS) * 0.3).astype(np.float32)
    sample, larger, largest = _sample(40, 20), _sample(80, 30), _sample(150, 40)
    want = B.Closure(theta).loss_grad(*sample, 1e-3)[1]
    cl = B.Closure(theta)
    if before:
        cl.loss_grad(*_sample(*before), 1e-3)
    grad = torch.zeros(B.CLOSURE_PARAMS, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        _grad_without_loss(cl, sample, grad)
    for other in (None, larger, largest):
        if other:
            cl.loss_grad(*other, 1e-3)
        grad.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(grad, want)
