"""The FP64 default's tables are made only where they are a small share of the
free device memory: with less than eight times their size left the mesh steps
on shape 1, which needs none, with the same bits; else on shape 7."""
import pytest

from paper_1408_5715_gb300 import binding as B
from paper_1408_5715_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def test_little_free_memory_keeps_the_tables_out():
    mi = W.periodic_square(1000, 800, seed=4)  # 1.6M cells: tables of some 120 MB
    m = B.Mesh.from_input(mi, "f64")
    perm = m.renumber("hilbert")
    U0 = torch.tensor(W.random_smooth_state(mi.centroids(), 1)[perm], device="cuda")
    V, U = U0.clone(), U0.clone()
    m.upload()
    torch.cuda.synchronize()
    taken = torch.empty(torch.cuda.mem_get_info()[0] - 800 * 2 ** 20, dtype=torch.uint8,
                        device="cuda")
    t = m.step(U, 3, 0.4)
    kernel = m.step_kernel()[0]
    left = torch.cuda.mem_get_info()[0]
    del taken
    torch.cuda.empty_cache()
    assert kernel == 1 and left >= 700 * 2 ** 20
    m.renumber("identity")  # the choice is made anew with the device arrays
    assert m.step(V, 3, 0.4) == t and m.step_kernel()[0] == 7
    assert torch.equal(U, V)
    m.close()
