"""Loss and gradient of the closure at the sizes where the gradient kernel's
16-row tiles and warps of 32 cells change (a few cells, one partial warp, one
cell more, several warps and blocks; walls, far field and periodic seams),
against the oracle's FP64 backward on inputs without ambiguous roundings, as
test_gpu_closure.py derives them and their tolerances; and one mesh after
another through one closure, whose scratch grows."""
import numpy as np
import pytest

from paper_1408_5715_gb300 import binding as B
from paper_1408_5715_gb300 import workloads as W
from test_gpu_closure import (SETTLED_WIDTH, make_theta, random_states, redraw_ambiguous_cells)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def closure():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return B.Closure(make_theta(8, scale=0.4)[0])


@pytest.mark.parametrize("kind,nx,ny", [("channel", 2, 2), ("channel", 4, 4), ("channel", 11, 3),
                                        ("square", 4, 3), ("square", 11, 3), ("square", 17, 15)])
def test_gradient_at_tile_edges(orc, closure, kind, nx, ny):
    prim = W.freestream(0.5)
    if kind == "channel":
        mi = W.channel_bump(nx, ny, seed=12)
        om_args = (mi.xy, mi.tri, None, mi.bnd, 0, W.conserved(*prim))
    else:
        mi = W.periodic_square(nx, ny, seed=12)
        om_args = (mi.xy, mi.tri, mi.canon, None, 0)
    rng = np.random.default_rng(nx * 100 + ny)
    _, th64 = make_theta(8, scale=0.4)
    om = orc.Mesh(*om_args)
    U0 = redraw_ambiguous_cells(om, random_states(rng, mi.n_tri), th64, rng)
    lo_s, hi_s, _ = om.closure_scale_intervals(U0, th64)
    assert (hi_s - lo_s).max() <= SETTLED_WIDTH
    Ut = (U0 + 0.02 * rng.normal(size=U0.shape)).astype(np.float32).astype(np.float64)
    dt, w = 2e-3, np.array([1.0, 0.5, 0.5, 2.0])
    g = B.Mesh.from_input(mi, "f32")
    g.set_freestream(*prim)
    Ud, Utd = (torch.tensor(x, dtype=torch.float32, device="cuda") for x in (U0, Ut))
    loss, grad = closure.loss_grad(g, Ud, Utd, dt, w)
    lo, go = om.closure_loss_grad(U0, Ut, dt, w, th64, bf16_acts=True)
    assert loss == pytest.approx(lo, rel=1e-5)
    grad = grad.cpu().numpy().astype(np.float64)
    for sl in (slice(0, 256), slice(256, 288), slice(288, 1312), slice(1312, 1344),
               slice(1344, 1376), slice(1376, 1377)):
        assert np.linalg.norm(grad[sl] - go[sl]) <= 1e-3 * np.linalg.norm(go[sl]), sl
        assert (np.abs(grad[sl] - go[sl]) <= 1e-3 * np.abs(go[sl]).max()).all(), sl
