"""fv_step in a CUDA graph that the caller captures, on meshes without a chosen
shape: the graph's steps need none of the tables of the default paths, so it
replays the bits of a direct call, before and after shapes, tile sizes and the
autotuner replaced those tables."""
import pytest

from paper_1408_5715_gb300 import binding as B
from paper_1408_5715_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("prec,nx,ny,default,captured", [
    ("f32", 64, 32, B.KERNEL_LOOP, 0), ("f32", 150, 100, B.KERNEL_ONE_WAVE, 0),
    ("f32", 480, 250, 1, 1), ("f64", 100, 60, 7, 1)])
@pytest.mark.parametrize("first", ["stepped", "uploaded"])
def test_captured_steps_outlive_the_tables(prec, nx, ny, default, captured, first):
    mi = W.periodic_square(nx, ny, seed=4)
    m = B.Mesh.from_input(mi, prec)
    perm = m.renumber("hilbert")
    U0 = torch.tensor(W.random_smooth_state(mi.centroids(), 1)[perm], dtype=m.torch_dtype,
                      device="cuda")
    m.upload()
    want = U0.clone()
    if first == "stepped":
        m.step(want, 5, 0.4)
        assert m.step_kernel()[0] == default
    U = U0.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        m.step(U, 5, 0.4, sync=False)
    assert m.step_kernel() == (captured, 0)
    if first == "uploaded":
        m.step(want, 5, 0.4)
    assert m.step_kernel()[0] == (default if first == "uploaded" else captured)

    def replay():
        U.copy_(U0)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(U, want)

    replay()
    for shape, tile in ((6, 96), (7, 200), (6, 0)):
        m.set_variant(shape)
        m.set_blocking(1, tile)
        m.step(U0.clone(), 3, 0.4)
        replay()
    m.autotune(U0)
    m.step(U0.clone(), 3, 0.4)
    replay()
    m.close()
