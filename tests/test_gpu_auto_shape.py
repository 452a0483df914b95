"""The kernel shape the library takes when none was chosen (by precision, size
and order of the mesh) against one thread per cell: the same bits, on both
sides of every line of the rule and for orders whose tiles are not compact."""
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


CASES = [
    ("f32", 97, 64, "hilbert"),    # 12,416 cells: the first that one cluster does not hold
    ("f32", 150, 100, "rcm"),      # long rings
    ("f32", 150, 100, "shuffle"),  # every neighbour in another tile: no tiles
    ("f32", 300, 150, "hilbert"),  # 90,000: the last of the one-wave tiles
    ("f32", 301, 150, "hilbert"),  # shape 0
    ("f32", 480, 240, "am1"),      # 230,400: shape 1
    ("f64", 5, 4, None),           # one small tile
    ("f64", 64, 31, "hilbert"),
    ("f64", 150, 100, "rcm"),
    ("f64", 150, 100, "shuffle"),
    ("f64", 230, 150, "am1"),
]


@pytest.mark.parametrize("prec,nx,ny,order", CASES)
def test_default_shape_is_bitwise_one_thread_per_cell(prec, nx, ny, order):
    mi = W.channel_bump(nx, ny, seed=4)
    prim = W.freestream(0.5)
    U0 = W.random_smooth_state(mi.centroids(), 2)
    for scheme, wave, steps, cfl in (("fe", "average", 101, 0.3), ("rk2", "max", 7, 0.3),
                                     ("fe", "average", 5, -1e-6)):
        got = []
        for shape in (None, 0):
            m = B.Mesh.from_input(mi, prec)
            m.set_freestream(*prim)
            perm = m.renumber(order, seed=3) if order else np.arange(mi.n_tri)
            m.set_wave_speed(wave)
            if shape is not None:
                m.set_variant(shape)
            else:
                m.upload()
                assert m.tiling() == (1, 1024)  # what the mesh reports is unchanged
            U = torch.tensor(U0[perm], dtype=m.torch_dtype, device="cuda")
            got.append((m.step(U, steps, cfl, scheme=scheme), U))
            m.close()
        assert torch.isfinite(got[0][1]).all()
        assert got[0][0] == got[1][0]
        assert torch.equal(got[0][1], got[1][1])


def test_shapes_chosen_later_and_earlier():
    """The library's choice gives way to a later one, and two steps per launch,
    a closure and a new order work after it."""
    mi = W.channel_bump(150, 100, seed=4)
    U0 = W.uniform_state(mi.n_tri, W.freestream(0.5))
    ref = None
    for later in ("none", "variant", "tile", "pairs", "back"):
        m = B.Mesh.from_input(mi, "f32")
        m.set_freestream(*W.freestream(0.5))
        m.upload()
        m.renumber("shuffle", seed=1)
        U = torch.tensor(U0, dtype=torch.float32, device="cuda")
        m.step(U, 2, -1e-5)
        perm = m.renumber("hilbert")  # the state is uniform up to the wall cells' change
        U = U[torch.tensor(perm, device="cuda").long()].contiguous()
        if later == "variant":
            m.set_variant(6)
        elif later == "tile":
            m.set_variant(7)
            m.set_blocking(1, 96)
        elif later == "pairs":
            m.set_blocking(2, 512)
        elif later == "back":
            m.set_blocking(2, 512)
            m.step(U.clone(), 4, -1e-5)
            m.set_blocking(1)
        m.step(U, 6, -1e-5)
        ref = U if ref is None else ref
        assert torch.equal(U, ref), later
        m.close()
