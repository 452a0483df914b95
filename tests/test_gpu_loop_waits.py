"""Waits of the resident loop that run out: at a limit of 0 every wait gives up
and the call returns FV_ETIMEOUT; at small limits some do, on some blocks, with
stores on their way (then FV_ETIMEOUT, else the right bits).  Afterwards the
mesh steps on from a good state, bit for bit, with the default limit."""
import pytest

from paper_1408_5715_gb300 import binding as B
from paper_1408_5715_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("scheme,blocking,comp", [("fe", 1, True), ("fe", 2, False),
                                                  ("rk2", 1, True)])
@pytest.mark.parametrize("nx,ny", [(8, 4), (60, 40), (96, 64)])  # 1 and 16 blocks
def test_waits_that_run_out(scheme, blocking, comp, nx, ny):
    mi = W.periodic_square(nx, ny, seed=3)
    m = B.Mesh.from_input(mi, "f32")
    perm = m.renumber("hilbert")
    m.set_compensation(comp)
    m.set_blocking(blocking)
    U0 = torch.tensor(W.random_smooth_state(mi.centroids(), 1)[perm], dtype=torch.float32,
                      device="cuda")

    def run(steps):
        U = U0.clone()
        return m.step(U, steps, 0.4, scheme=scheme), U

    good = {steps: run(steps) for steps in (1, 40)}
    for limit in (0, 0, 1, 2, 3, 5, 8, 16, 64, 1024):
        m.set_wait_limit(limit)
        for steps in (40, 1):
            try:
                t, U = run(steps)
                assert limit > 0
                assert t == good[steps][0] and torch.equal(U, good[steps][1])
            except B.FVError as e:
                assert e.code == B.FV_ETIMEOUT
    m.set_wait_limit(1 << 24)
    for steps in (1, 40):
        t, U = run(steps)
        assert t == good[steps][0] and torch.equal(U, good[steps][1])
    m.close()
