"""The batch's default shape on both sides of its lines: one thread per cell,
and tiles for FP64 above 200,000 cells and the compensated update above two
million; the same bits as the other shape."""
import pytest

from paper_1408_5715_gb300 import binding as B
from paper_1408_5715_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("prec,n,want", [("f32", 550, {True: 0, False: 0}),
                                         ("f32", 600, {True: 6, False: 0}),
                                         ("f64", 180, {None: 0}), ("f64", 190, {None: 6})])
def test_default_shape_by_size_and_update(prec, n, want):
    mi = W.periodic_square(n, n, seed=3)  # three of them
    U0 = W.isentropic_vortex(mi.centroids())
    meshes = [B.Mesh.from_input(mi, prec) for _ in range(3)]
    perms = [m.renumber("hilbert") for m in meshes]
    b = B.Batch(meshes)
    U0 = torch.tensor(b.pack([U0[p] for p in perms]), dtype=b.torch_dtype, device="cuda")
    got = {}
    for comp, shape in want.items():
        if comp is not None:
            b.set_compensation(comp)
        U = U0.clone()
        got[comp] = (b.step(U, 4, 0.4), U)
        assert b.step_kernel() == shape and b.variant() == 6
    for comp, shape in want.items():
        if comp is not None:
            b.set_compensation(comp)
        b.set_variant(6 - shape)
        U = U0.clone()
        assert (b.step(U, 4, 0.4) == got[comp][0]).all() and torch.equal(U, got[comp][1])
        assert b.step_kernel() == 6 - shape
