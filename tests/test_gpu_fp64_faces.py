"""FP64: shape 7 (each face once, the CFL bound ruled out in FP32) against one
thread per cell, bit for bit, at the tile sizes where its blocks change and on
states where the FP32 bound decides nothing; and the FP64 reciprocal and square
root, seen through the CFL step, against extended precision."""
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


def _state(kind, c, rng):
    if kind == "smooth":
        return W.random_smooth_state(c, 3)
    if kind == "uniform":  # every cell may hold the minimum
        return W.uniform_state(len(c), W.freestream(0.5))
    if kind == "fast":  # internal energy below 1 % of the total: no FP32 bound
        return W.uniform_state(len(c), W.freestream(25.0)) * (1 + 1e-3 * rng.random((len(c), 1)))
    scale = 10.0 ** rng.uniform(-40, 40)  # outside the quick range of recip and root
    return W.random_smooth_state(c, 4) * scale


def _run(mi, U0, prim, shape, tile, scheme, wave, cfl, steps=7):
    m = B.Mesh.from_input(mi, "f64")
    m.set_freestream(*prim)
    perm = m.renumber("hilbert")
    m.set_wave_speed(wave)
    m.set_variant(shape)
    if tile:
        m.set_blocking(1, tile)
    U = torch.tensor(U0[perm], dtype=torch.float64, device="cuda")
    t = m.step(U, steps, cfl, scheme=scheme)
    m.close()
    return t, U


@pytest.mark.parametrize("state", ["smooth", "uniform", "fast", "scaled"])
@pytest.mark.parametrize("tile", [32, 64, 65, 128, 129, 384, 513, 800])
def test_shape_7_is_bitwise_one_thread_per_cell(state, tile):
    rng = np.random.default_rng(tile)
    for mi, prim in ((W.periodic_square(37, 23, seed=5), (1.0, 0.0, 0.0, 1.0)),
                     (W.channel_bump(40, 17, seed=5), W.freestream(0.5))):
        if state == "fast" and prim[1]:
            continue  # no flow over the bump at this speed stays positive
        U0 = _state(state, mi.centroids(), rng)
        for scheme, wave in (("fe", "average"), ("rk2", "max")):
            cfl = 0.02 if state == "fast" else 0.2
            ref = _run(mi, U0, prim, 0, 0, scheme, wave, cfl)
            got = _run(mi, U0, prim, 7, tile, scheme, wave, cfl)
            assert torch.isfinite(got[1]).all() and got[0] == ref[0] > 0
            assert torch.equal(got[1], ref[1])


@pytest.mark.parametrize("bad", ["nan", "inf", "rho", "p"])
def test_shape_7_reports_a_bad_state(bad):
    mi = W.periodic_square(37, 23, seed=5)
    U0 = W.random_smooth_state(mi.centroids(), 3)
    m = B.Mesh.from_input(mi, "f64")
    m.set_variant(7)
    m.set_blocking(1, 128)
    U0[700, 0 if bad == "rho" else 3] = {"nan": np.nan, "inf": np.inf, "rho": -1.0, "p": 1e-3}[bad]
    U = torch.tensor(U0, dtype=torch.float64, device="cuda")
    with pytest.raises(B.FVError) as e:
        m.step(U, 2, -1e-9)
    assert e.value.code == B.FV_ENONFINITE


def test_fp64_reciprocal_and_root_against_extended_precision():
    """dt of two cells = the smaller 2V / (P (|v| + c)).  Its 15 FP64 operations
    (two reciprocals, two square roots) on the state, each within 0.51 ulp, on
    top of the rounding of 2V / P, stay within 16 ulp of extended precision."""
    if np.finfo(np.longdouble).eps > 1e-18:
        pytest.skip("no extended precision")
    rng = np.random.default_rng(8)
    mi = W.two_cells()
    m = B.Mesh.from_input(mi, "f64")
    ld = np.longdouble
    worst = 0.0
    for k in range(400):
        rho, p = 10.0 ** rng.uniform(-3, 3, 2)
        u, v = rng.normal(size=2) * np.sqrt(p / rho)
        U0 = W.conserved(rho, u, v, p)
        if k % 4 == 0:
            U0 = U0 * 10.0 ** rng.uniform(-45, 45)
        r, mx, my, E = (ld(x) for x in U0)
        # gamma and gamma - 1 as the kernels hold them
        pp = ld(1.4 - 1.0) * (E - (mx * mx + my * my) / (2 * r))
        c = np.sqrt(ld(1.4) * pp / r)
        lam = np.sqrt((mx / r) ** 2 + (my / r) ** 2) + c
        want = ld(1.0) / (2 + np.sqrt(ld(2))) / lam
        U = torch.tensor(np.repeat(U0[None], 2, 0), dtype=torch.float64, device="cuda")
        got = m.compute_dt(U, 1.0)
        # the pressure's cancellation magnifies the rounding of its terms
        cond = float((E + (mx * mx + my * my) / (2 * r)) * ld(1.4 - 1.0) / pp)
        worst = max(worst, abs(float((ld(got) - want) / want)) / (2.2e-16 * max(cond, 1.0)))
    assert worst <= 8.0, worst
