"""Float-float and difference sums with one query per CTA: sizes at the edges of its rows (128
pixels), tiles (256), row ranges and item queue (a single query, few queries split over many row
ranges, more queries than items per CTA), against the FP64 oracle with the gates of
test_gpu_ff.py (1e-11 of the absolute-value sums) and test_gpu_difference.py (the library's own
bound)."""
import numpy as np
import pytest

import oracle
from gates import abs_scales, oracle_boundary
from test_gpu_difference import _difference_case
from test_gpu_eval import random_mag, random_points, run_eval

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [(1, 1, 1), (16, 8, 3), (43, 3, 2), (16, 16, 129), (257, 1, 33), (19, 27, 6500),
         (128, 70, 1), (90, 91, 13)]


@pytest.fixture(scope="module")
def dbie():
    import paper_1306_1122_gb300 as d
    return d


@pytest.mark.parametrize("nx,ny,n", SIZES)
def test_float_float_sizes(dbie, nx, ny, n):
    mag = random_mag(nx, ny, 300 + nx)
    xyz, lam = random_points(mag, n, 301 + n, zlo=0.3, zhi=25.0)
    got = run_eval(dbie, mag, xyz, lam, dbie._native.DBIE_PREC_FLOAT_FLOAT)
    B, G, _ = oracle.field(oracle_boundary(mag), xyz.astype(np.float64), lam.astype(np.float64))
    sB, sG = abs_scales(mag, xyz, lam)
    assert np.all(np.abs(got["B"] - B) <= 1e-11 * sB)
    assert np.all(np.abs(got["gradB"] - G) <= 1e-11 * sG[:, :, None])


@pytest.mark.parametrize("tied", [False, True])
@pytest.mark.parametrize("nx,ny,n", SIZES)
def test_difference_sizes(dbie, nx, ny, n, tied):
    mag = random_mag(nx, ny, 310 + nx)
    xyz, lam0 = random_points(mag, n, 311 + n, zlo=0.3, zhi=25.0)
    r = _difference_case(dbie, mag, xyz, lam0, 1e-3, tied, seed=n)
    assert np.all(r["errB"] <= r["bB"]) and np.all(r["errG"] <= r["bG"])
