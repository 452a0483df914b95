"""The closure's gradient under loss weights that scale it by powers of two: the
bits of the gradient at weight 1, scaled, in every component that is a normal
float (at 2^-88 the smallest of the cells' terms is 6e-36) -- no operand of the
tensor cores loses bits to its size.  Components that come out subnormal are off
by half their spacing, 2^-150, at most."""
import numpy as np
import pytest

from paper_1408_5715_gb300 import binding as B
from paper_1408_5715_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("power", [-35, -10, 20, 38, 44])
def test_gradient_scales_with_the_weights(power):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    mi = W.channel_bump(40, 20, seed=2)
    m = B.Mesh.from_input(mi, "f32")
    rng = np.random.default_rng(1)
    U = W.random_smooth_state(mi.centroids(), 1)
    U0, Ut = (torch.tensor(x, dtype=torch.float32, device="cuda")
              for x in (U, U * (1 + 0.1 * rng.normal(size=U.shape))))
    cl = B.Closure((rng.normal(size=B.CLOSURE_PARAMS) * 0.3).astype(np.float32))
    loss1, grad1 = cl.loss_grad(m, U0, Ut, 1e-3)
    for _ in range(2):  # and the scratch is at rest again after a call
        loss, grad = cl.loss_grad(m, U0, Ut, 1e-3, weights=(2.0 ** power,) * 4)
        assert loss == loss1 * 4.0 ** -power
        got, want = grad.double() * 4.0 ** power, grad1.double()
        normal = want.abs() >= 2.0 ** -126 * 4.0 ** power
        assert torch.equal(got[normal], want[normal]) and normal.sum() > 500
        assert ((got - want).abs() <= 2.0 ** -150 * 4.0 ** power)[~normal].all()
    assert torch.equal(cl.loss_grad(m, U0, Ut, 1e-3)[1], grad1)
