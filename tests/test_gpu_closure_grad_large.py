"""The closure's gradient on meshes of more cells than the gradient kernel's
resident blocks take at a time (128 a block, three blocks an SM: 58,368 on 152
SMs): warps go on to further cells and carry rows of an unfinished tile with
them.  Against the oracle's FP64 backward, with the tolerances of
test_gpu_closure_grad.py."""
import numpy as np
import pytest

from paper_1408_5715_gb300 import binding as B
from paper_1408_5715_gb300 import workloads as W
from test_gpu_closure import (SETTLED_WIDTH, make_theta, random_states, redraw_ambiguous_cells)

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nx,ny", [(211, 151), (389, 160)])  # 63,722 and 124,480 cells
def test_gradient_beyond_the_resident_warps(orc, nx, ny):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    prim = W.freestream(0.5)
    mi = W.channel_bump(nx, ny, seed=12)
    om = orc.Mesh(mi.xy, mi.tri, None, mi.bnd, 0, W.conserved(*prim))
    rng = np.random.default_rng(nx)
    th, th64 = make_theta(8, scale=0.4)
    U0 = redraw_ambiguous_cells(om, random_states(rng, mi.n_tri), th64, rng)
    lo_s, hi_s, _ = om.closure_scale_intervals(U0, th64)
    assert (hi_s - lo_s).max() <= SETTLED_WIDTH
    Ut = (U0 + 0.02 * rng.normal(size=U0.shape)).astype(np.float32).astype(np.float64)
    dt, w = 2e-3, np.array([1.0, 0.5, 0.5, 2.0])
    g = B.Mesh.from_input(mi, "f32")
    g.set_freestream(*prim)
    Ud, Utd = (torch.tensor(x, dtype=torch.float32, device="cuda") for x in (U0, Ut))
    loss, grad = B.Closure(th).loss_grad(g, Ud, Utd, dt, w)
    lo, go = om.closure_loss_grad(U0, Ut, dt, w, th64, bf16_acts=True)
    assert loss == pytest.approx(lo, rel=1e-5)
    grad = grad.cpu().numpy().astype(np.float64)
    for sl in (slice(0, 256), slice(256, 288), slice(288, 1312), slice(1312, 1344),
               slice(1344, 1376), slice(1376, 1377)):
        assert np.linalg.norm(grad[sl] - go[sl]) <= 1e-3 * np.linalg.norm(go[sl]), sl
        assert (np.abs(grad[sl] - go[sl]) <= 1e-3 * np.abs(go[sl]).max()).all(), sl
