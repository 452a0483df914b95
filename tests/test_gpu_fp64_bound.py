"""The CFL minimum of shape 7 in FP64, which rules cells out by an FP32 bound,
against one thread per cell on states whose speeds overflow or vanish in FP32
while density, energy and pressure are ordinary numbers: the same time, bit for
bit.  The cell of the smallest bound is the slower one, so that a bound lost in
FP32 shows."""
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


def _graded_strip():
    mi = W.shock_tube_strip(64, 8, seed=3)
    mi.xy[:, 0] = 0.05 * mi.xy[:, 0] + mi.xy[:, 0] ** 2  # the cells on the left are the smallest
    return mi


# density, internal energy in the small cells and in the others, velocity
CASES = [
    (1e-19, 5e19, 9e19, 0.0),      # sound speed squared above the largest float
    (1e-19, 5e19, 9e19, 1e18),
    (2e-20, 2e18, 2e18, 2e19),     # velocity squared above it
    (1e18, 2.3e-20, 1.9e-20, 0.0),  # sound speed squared below the smallest normal float
    (1e18, 1.9e-20, 2.3e-20, 0.0),
    (9e19, 1.1e-20, 1.2e-20, 0.0),
    (1e-19, 5e-5, 9e-5, 0.0),      # ordinary speeds for comparison
]


@pytest.mark.parametrize("rho,e_small,e_large,u", CASES)
@pytest.mark.parametrize("scale", [1e-19, 1.0, 1e19])
def test_minimum_at_speeds_outside_the_float_range(rho, e_small, e_large, u, scale):
    mi = _graded_strip()
    small = mi.centroids()[:, 0] < np.median(mi.centroids()[:, 0])
    U0 = np.zeros((mi.n_tri, 4))
    U0[:, 0] = rho
    U0[:, 1] = rho * u
    U0[:, 3] = np.where(small, e_small, e_large) + 0.5 * rho * u * u
    mi.xy[:] *= scale  # the inradii's range too
    got = []
    for shape in (0, 7):
        m = B.Mesh.from_input(mi, "f64")
        m.set_variant(shape)
        m.set_blocking(1, 128)
        U = torch.tensor(U0, dtype=torch.float64, device="cuda")
        t = [m.step(U, steps, 1e-3) for steps in (1, 2, 5)]
        assert t[-1] > 0 and torch.isfinite(U).all()
        got.append((t, U))
        m.close()
    assert got[0][0] == got[1][0]
    assert torch.equal(got[0][1], got[1][1])
