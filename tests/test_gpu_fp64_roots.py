"""The FP64 reciprocal and square root of the kernels (cell_math.cuh), compiled
as they stand, against the correctly rounded operations: equal outside the range
in which they start from FP32, within 0.5 + 2^-9 ulp of the exact value inside.

The bound: the FP32 start is good to 2^-21 (2^-22.4 for the inverse root, plus
2^-23 for the truncated argument).  The reciprocal's third-order step leaves the
cube of that, 2^-63, which is 2^-10 ulp; the root's second step leaves a product
of the first step's error (1.5 times the square, below 2^-41) and the start's,
below 2^-62: 2^-9 ulp.  The last operation rounds once.  A result that differs
from the correctly rounded one therefore lies within 2^-9 ulp of a tie, and at
most one in 2^-8 does."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1408_5715_gb300 import build as BLD

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def roots(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    out = str(tmp_path_factory.mktemp("roots") / "fp64_roots.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "fp64_roots.cu")
    subprocess.run([BLD.nvcc(), "-shared", "-o", out, src] + BLD._flags(src), check=True,
                   capture_output=True)
    lib = ctypes.CDLL(out)
    lib.fp64_roots.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int, ctypes.c_void_p]

    def run(x):
        d = torch.tensor(x, device="cuda")
        r, s = torch.empty_like(d), torch.empty_like(d)
        stream = torch.cuda.current_stream().cuda_stream
        assert lib.fp64_roots(d.data_ptr(), r.data_ptr(), s.data_ptr(), d.numel(), stream) == 0
        return r.cpu().numpy(), s.cpu().numpy()

    return run


def test_the_correctly_rounded_operations_outside_the_quick_range(roots):
    rng = np.random.default_rng(1)
    lo, hi = 2.0 ** -100, 2.0 ** 100
    x = np.concatenate([
        [0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 1e-310, 1.7e308, -1.0, -1e-200, hi,
         np.nextafter(lo, 0), np.nextafter(hi, np.inf)],
        10.0 ** rng.uniform(-307, -31, 5000), 10.0 ** rng.uniform(31, 307, 5000),
        -(10.0 ** rng.uniform(-307, 307, 5000))])
    r, s = roots(x)
    with np.errstate(all="ignore"):
        assert np.array_equal(r, 1.0 / x, equal_nan=True)
        assert np.array_equal(s, np.sqrt(x), equal_nan=True)


def test_bound_inside_the_quick_range(roots):
    if np.finfo(np.longdouble).eps > 1e-18:
        pytest.skip("no extended precision")
    rng = np.random.default_rng(2)
    lo, hi = 2.0 ** -100, 2.0 ** 100
    x = np.concatenate([
        2.0 ** rng.integers(-100, 100, 200).astype(float),
        [lo, np.nextafter(lo, 1), np.nextafter(hi, 0), 1.0, np.nextafter(1, 0), np.nextafter(1, 2)],
        rng.uniform(1.0, 4.0, 60000), 2.0 ** rng.uniform(-100, 100, 60000)])
    ld = np.longdouble
    xl = x.astype(ld)
    # what extended precision itself rounds (2^-11 ulp of FP64 where it has 64 bits)
    slack = 2.0 ** -9 + float(np.finfo(ld).eps) / 2.0 ** -52
    for got, want, rounded in zip(roots(x), (ld(1) / xl, np.sqrt(xl)), (1.0 / x, np.sqrt(x))):
        ulp = np.spacing(np.minimum(got, rounded))
        assert (np.abs(got.astype(ld) - want) <= (0.5 + slack) * ulp).all()
        assert (got == rounded).mean() >= 1.0 - 2.0 ** -8
