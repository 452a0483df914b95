"""The resident loop in launches of one CFL bound (one step, or two that share
it) whose dt t_stop clamps: every block forms it from the time the launch
started at.  Against a launch per step, bit for bit, over many launches."""
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


@pytest.mark.parametrize("steps", [1, 2])
@pytest.mark.parametrize("share", [0.3, 0.999, 1.5])
def test_clamped_launches_of_one_bound(steps, share):
    mi = W.periodic_square(96, 64, seed=3)  # 12,288 cells on 16 blocks
    U0 = W.random_smooth_state(mi.centroids(), 1)
    got = []
    for chosen in (False, True):
        m = B.Mesh.from_input(mi, "f32")
        perm = m.renumber("hilbert")
        if steps == 2:
            m.set_blocking(2, 1024 if chosen else 0)
        elif chosen:
            m.set_variant(0)
        U = torch.tensor(U0[perm], dtype=torch.float32, device="cuda")
        t_stop = share * steps * m.compute_dt(U, 0.4)
        got.append(([m.step(U, steps, 0.4, t_stop=t_stop) for _ in range(50)], U))
        m.close()
    assert got[0][0] == got[1][0] and got[0][0][0] > 0
    assert torch.equal(got[0][1], got[1][1])
