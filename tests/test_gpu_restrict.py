"""Restriction by area-weighted means over its forms: ids read one at a time
and four at a time (numbers of children, unaligned ids), FP32 and FP64 on both
sides, coarse counts around the block size, and area sums outside the range in
which a float result is formed with a reciprocal, down to subnormal areas;
against FP64 sums on the host."""
import numpy as np
import pytest

from paper_1408_5715_gb300 import binding as B

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("fine", ["f32", "f64"])
@pytest.mark.parametrize("coarse", ["f32", "f64"])
@pytest.mark.parametrize("kids,offset", [(1, 0), (3, 0), (4, 0), (4, 1), (6, 0), (16, 0), (16, 3)])
@pytest.mark.parametrize("scale", [1.0, 1e-40, 1e-310, 1e300])
def test_means_of_every_form(fine, coarse, kids, offset, scale):
    dt = {"f32": torch.float32, "f64": torch.float64}
    rng = np.random.default_rng(kids)
    for n in (1, 255, 300):
        nf = n * kids
        U = torch.tensor(rng.normal(size=(nf, 4)) + 0.5, device="cuda").to(dt[fine])
        area = rng.uniform(0.5, 1.5, nf) * scale
        ids = rng.permutation(nf).reshape(n, kids)
        flat = torch.zeros(nf + offset, dtype=torch.int32, device="cuda")
        flat[offset:] = torch.tensor(ids.reshape(-1).astype(np.int32), device="cuda")
        out = torch.full((n, 4), float("nan"), dtype=dt[coarse], device="cuda")
        B.restrict_mean(U, torch.tensor(area, device="cuda"), flat[offset:].reshape(n, kids), out)
        u = U.double().cpu().numpy()[ids]
        w = (area / scale)[ids][..., None]
        want = (w * u).sum(1) / w.sum(1)
        mag = (w * np.abs(u)).sum(1) / w.sum(1)
        # relative: rounding of sums, quotient and result; absolute, on subnormal
        # sums: 2^-1075 for each of the products over at least 5e-311 each
        tol = (2.0 ** -24 if coarse == "f32" else 0.0) + (2 * kids + 6) * 2.0 ** -53
        lost = 2.0 ** -1074 / 5e-311 / 2 if scale == 1e-310 else 0.0
        got = out.double().cpu().numpy()
        assert (np.abs(got - want) <= tol * mag + lost).all()
