"""The tables of the default paths: built by the first step that runs them (a
mesh that is only monitored holds its own arrays and no more), and there again
after two steps per launch or another tile size had the mesh in between."""
import pytest

from paper_1408_5715_gb300 import binding as B
from paper_1408_5715_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _mesh(prec, nx, ny):
    mi = W.periodic_square(nx, ny, seed=4)
    m = B.Mesh.from_input(mi, prec)
    perm = m.renumber("hilbert")
    U = torch.tensor(W.random_smooth_state(mi.centroids(), 1)[perm], dtype=m.torch_dtype,
                     device="cuda")
    return m, U, torch.empty_like(U)


def test_a_monitored_mesh_holds_no_tables():
    def monitor(m, U, R):
        m.upload()
        m.compute_dt(U, 0.4)
        m.residual(U, out=R)
        m.totals(U)

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    monitor(*_mesh("f64", 20, 10))  # the device code is loaded
    m, U, R = _mesh("f64", 600, 500)
    before = free()
    monitor(m, U, R)
    # neighbours 16, geometry 64, area 8, work 32 bytes a cell, each in pages of 2 MB
    assert before - free() <= 120 * m.n + 16 * 2 ** 20
    m.step(U, 2, 0.4)
    assert m.step_kernel()[0] == 7
    m.close()


@pytest.mark.parametrize("nx,ny,want", [(64, 32, B.KERNEL_LOOP), (150, 100, B.KERNEL_ONE_WAVE),
                                        (400, 250, 0)])
@pytest.mark.parametrize("between", ["uploaded", "stepped"])
def test_default_after_two_steps_per_launch(nx, ny, want, between):
    m, U, _ = _mesh("f32", nx, ny)
    V = U.clone()
    m.set_blocking(2, 512)
    m.upload()
    if between == "stepped":
        m.step(U, 4, -1e-5)
        assert m.step_kernel() == (B.KERNEL_PAIRS, 512)
        U.copy_(V)
    m.set_blocking(1)
    t = m.step(U, 5, 0.4)
    assert m.step_kernel()[0] == want
    m.set_variant(0)
    assert m.step(V, 5, 0.4) == t and torch.equal(U, V)
    m.close()
