"""The resident loop (a whole time loop in one launch, csrc/loop_step.cu)
against a launch per step: the same bits in state, time and remainder, over
both schemes, updates, wave speeds, boundary kinds, orders and the sizes
where its tiles change (one block, block sizes, partial last tiles, the
largest mesh it takes, several launches)."""
import numpy as np
import pytest

from paper_1408_5715_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_mod():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    return torch


def _mesh(kind, nx, ny):
    if kind == "square":
        mi = W.periodic_square(nx, ny, seed=3)
        return mi, W.random_smooth_state(mi.centroids(), 1), (1.0, 0.0, 0.0, 1.0)
    if kind == "channel":
        mi = W.channel_bump(nx, ny, seed=3)
        prim = W.freestream(0.5)
        return mi, W.uniform_state(mi.n_tri, prim), prim
    if kind == "strip":
        mi = W.shock_tube_strip(nx, ny, seed=3)
        return mi, W.sod_state(mi.centroids()), (1.0, 0.0, 0.0, 1.0)
    mi = W.forward_step(nx // 4, nx - nx // 4, ny // 4, ny - ny // 4, seed=3)
    prim = W.mach3_inflow()
    return mi, W.uniform_state(mi.n_tri, prim), prim


def _run(torch, B, mi, U0, prim, order, steps, cfl, shape=None, comp=True, scheme="fe",
         wave="average", blocking=None, t_stop=0.0, remainder=False, calls=1):
    m = B.Mesh.from_input(mi, "f32")
    m.set_freestream(*prim)
    perm = m.renumber(order) if order else np.arange(mi.n_tri)
    m.set_compensation(comp)
    m.set_wave_speed(wave)
    if blocking:
        m.set_blocking(*blocking)
    if shape is not None:
        m.set_variant(shape)
    U = torch.tensor(U0[perm], dtype=torch.float32, device="cuda")
    lo = torch.zeros((m.n, 4), dtype=torch.int16, device="cuda")
    if remainder:
        m.set_remainder(lo)
    t = [m.step(U, steps, cfl, t_stop=t_stop, scheme=scheme) for _ in range(calls)]
    m.close()
    return U.cpu().numpy(), t, lo.cpu().numpy()


CASES = [
    ("square", 8, 4, "hilbert", 7, {}),                       # one block, no ring
    ("square", 10, 7, None, 5, dict(comp=False)),             # 140 cells: three tiles, one partial
    ("square", 64, 32, "rcm", 250, {}),                       # 16 tiles of 256, wide rings
    ("square", 64, 32, "shuffle", 20, dict(comp=False)),      # every neighbour in another tile
    ("square", 64, 32, "hilbert", 1, dict(remainder=True, calls=3)),
    ("square", 257, 8, "hilbert", 9, {}),                     # tiles of 257: 512-thread blocks
    ("strip", 603, 10, "hilbert", 60, dict(comp=False, scheme="rk2")),  # tiles of 754
    ("channel", 95, 53, "hilbert", 41, dict(scheme="rk2", remainder=True, calls=2)),
    ("channel", 100, 61, "hilbert", 40, dict(wave="max")),
    ("channel", 60, 30, "hilbert", 40, dict(wave="max", scheme="rk2", comp=False)),
    ("step", 70, 60, "hilbert", 60, {}),
    ("square", 64, 63, "hilbert", 30, dict(comp=False, t_stop=0.01)),
    ("square", 96, 64, "hilbert", 30, {}),                    # the largest: 12,288 cells
    ("square", 12, 10, "hilbert", 4100, {}),                  # two launches
]


@pytest.mark.parametrize("kind,nx,ny,order,steps,kw", CASES)
def test_resident_loop_is_bitwise_a_launch_per_step(torch_mod, kind, nx, ny, order, steps, kw):
    from paper_1408_5715_gb300 import binding as B
    mi, U0, prim = _mesh(kind, nx, ny)
    for cfl in (0.4, -1e-5):
        a = _run(torch_mod, B, mi, U0, prim, order, steps, cfl, **kw)
        b = _run(torch_mod, B, mi, U0, prim, order, steps, cfl, shape=0, **kw)
        assert np.isfinite(a[0]).all() and not np.array_equal(a[0], U0.astype(np.float32))
        assert a[1] == b[1]
        assert np.array_equal(a[0], b[0])
        assert np.array_equal(a[2], b[2])


@pytest.mark.parametrize("steps,comp", [(1, True), (8, False), (9, True), (101, False)])
def test_resident_loop_with_one_bound_per_two_steps(torch_mod, steps, comp):
    """Two steps per bound with the tile size left to the library against the
    two-step kernel on tiles of 1024 cells: dt from every second state."""
    from paper_1408_5715_gb300 import binding as B
    mi, U0, prim = _mesh("square", 61, 70)
    for cfl, t_stop in ((0.4, 0.0), (0.4, 0.004), (-1e-5, 0.0)):
        kw = dict(comp=comp, t_stop=t_stop, remainder=comp)
        a = _run(torch_mod, B, mi, U0, prim, "hilbert", steps, cfl, blocking=(2,), **kw)
        b = _run(torch_mod, B, mi, U0, prim, "hilbert", steps, cfl, blocking=(2, 1024), **kw)
        assert a[1] == b[1]
        assert np.array_equal(a[0], b[0])
        assert np.array_equal(a[2], b[2])


def test_resident_loop_reports_a_bad_state(torch_mod):
    from paper_1408_5715_gb300 import binding as B
    mi, U0, _ = _mesh("square", 64, 32)
    m = B.Mesh.from_input(mi, "f32")
    for bad in (np.nan, -1.0):
        U1 = U0.copy()
        U1[1000, 0] = bad
        U = torch_mod.tensor(U1, dtype=torch_mod.float32, device="cuda")
        with pytest.raises(B.FVError) as e:
            m.step(U, 3, 0.4)
        assert e.value.code == B.FV_ENONFINITE
    U = torch_mod.tensor(U0, dtype=torch_mod.float32, device="cuda")
    assert m.step(U, 3, 0.4) > 0  # and the mesh steps on from a good one
    m.close()
