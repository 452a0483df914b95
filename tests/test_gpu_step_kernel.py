"""What fv_step runs where no kernel shape was chosen, on each side of every
line of the rule, and after a choice: the bitwise tests of the default paths
would pass on a fallback too."""
import pytest

from paper_1408_5715_gb300 import binding as B
from paper_1408_5715_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _mesh(prec, nx, ny, order, kind="channel"):
    mi = W.channel_bump(nx, ny, seed=4) if kind == "channel" else W.periodic_square(nx, ny, seed=4)
    prim = W.freestream(0.5)
    m = B.Mesh.from_input(mi, prec)
    m.set_freestream(*prim)
    if order:
        m.renumber(order, seed=3)
    return m, torch.tensor(W.uniform_state(mi.n_tri, prim), dtype=m.torch_dtype, device="cuda")


DEFAULTS = [
    ("f32", 8, 4, None, 1, B.KERNEL_LOOP),
    ("f32", 96, 64, "hilbert", 1, B.KERNEL_LOOP),       # 12,288: the last on one cluster
    ("f32", 96, 64, "shuffle", 1, B.KERNEL_LOOP),
    ("f32", 96, 64, "hilbert", 2, B.KERNEL_LOOP),
    ("f32", 97, 64, "hilbert", 2, B.KERNEL_PAIRS),
    ("f32", 97, 64, "hilbert", 1, B.KERNEL_ONE_WAVE),
    ("f32", 150, 100, "shuffle", 1, 0),                 # no compact tiles
    ("f32", 300, 150, "hilbert", 1, B.KERNEL_ONE_WAVE),  # 90,000
    ("f32", 301, 150, "hilbert", 1, 0),
    ("f32", 460, 250, "hilbert", 1, 0),                 # 230,000
    ("f32", 480, 240, "hilbert", 1, 1),
    ("f64", 5, 4, None, 1, 7),
    ("f64", 230, 150, "hilbert", 1, 7),
    ("f64", 150, 100, "shuffle", 1, 1),
]


@pytest.mark.parametrize("prec,nx,ny,order,blocking,want", DEFAULTS)
def test_default_kernel(prec, nx, ny, order, blocking, want):
    m, U = _mesh(prec, nx, ny, order)
    assert m.step_kernel() == (-1, 0)
    if blocking == 2:
        m.set_blocking(2)
    m.upload()
    m.step(U, 0, -1e-6)
    assert m.step_kernel() == (-1, 0)
    m.step(U, 3, -1e-6)
    kernel, tile = m.step_kernel()
    assert kernel == want
    assert (tile > 0) == (want not in (0, 1))
    for shape in (6, 0):  # a choice is what runs from then on
        m.set_variant(shape)
        m.set_blocking(1, 256)
        m.step(U, 2, -1e-6)
        # tiles of 256 cells that are all resident at a time take the one-wave form
        assert m.step_kernel()[0] in ((6, B.KERNEL_ONE_WAVE) if shape == 6 else (0,))
    m.close()


def test_learned_kernels():
    m, U = _mesh("f32", 40, 20, "hilbert")
    cl = B.Closure()
    for shape, want in ((None, B.KERNEL_LEARNED), (7, B.KERNEL_LEARNED_TILES)):
        if shape:
            m.set_variant(shape)
        m.step(U, 2, -1e-6, closure=cl)
        assert m.step_kernel()[0] == want


def test_autotuned_kernel():
    m, U = _mesh("f32", 64, 32, "hilbert", "square")
    best, us = m.autotune(U)
    assert m.tiling()[0] == best and us[best] == min(us)
    m.step(U, 3, -1e-6)
    assert m.step_kernel()[0] == B.KERNEL_LOOP  # a third of any shape's time per step
    m, U = _mesh("f32", 300, 150, "hilbert")
    best, _ = m.autotune(U)
    m.step(U, 3, -1e-6)
    kernel, tile = m.step_kernel()
    assert kernel == best or (best == 6 and kernel == B.KERNEL_ONE_WAVE)
    assert best < 6 or tile == m.tiling()[1]


@pytest.mark.parametrize("prec,nx,count,want", [("f32", 60, 3, 0), ("f64", 60, 3, 0),
                                                ("f64", 200, 3, 6)])
def test_batch_kernel(prec, nx, count, want):
    mis = [W.periodic_square(nx, nx, seed=k) for k in range(count)]
    meshes = [B.Mesh.from_input(mi, prec) for mi in mis]
    for m in meshes:
        m.renumber("hilbert")
    b = B.Batch(meshes)
    assert b.step_kernel() == -1
    U = torch.tensor(b.pack([W.uniform_state(mi.n_tri, W.freestream(0.5)) for mi in mis]),
                     dtype=b.torch_dtype, device="cuda")
    b.step(U, 2, -1e-6)
    assert b.step_kernel() == want and b.variant() == 6
    b.set_variant(5)
    b.step(U, 2, -1e-6)
    assert b.step_kernel() == 5
