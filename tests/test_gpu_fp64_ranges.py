"""FP64 form over ranges of quarter tiles (64 pixels): boundaries that end inside, at and after a
quarter or a tile, with one query, a full block and a remainder, split to single quarters and not
split, against the oracle (1e-10 of the absolute-value sums, the FP64 form's gate)."""
import numpy as np
import pytest

import oracle
from gates import TOL_FP64, abs_scales, oracle_boundary
from test_gpu_eval import random_mag, random_points

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,n", [
    (1, 1, 1), (9, 7, 128), (16, 4, 129), (13, 5, 3), (16, 16, 1), (257, 1, 130), (23, 29, 40),
    (20, 16, 2600), (3, 2, 20011)])
def test_fp64_ranges(nx, ny, n):
    import paper_1306_1122_gb300 as dbie
    mag = random_mag(nx, ny, 40 + nx)
    xyz, lam = random_points(mag, n, 41 + n, zlo=0.3, zhi=9.0)
    f = dbie.DBIEField.from_magnetogram(mag)
    got = f.eval(torch.from_numpy(xyz), torch.from_numpy(lam), grad=True,
                 options=dbie.Options(precision=1))
    torch.cuda.synchronize()
    B, G, _ = oracle.field(oracle_boundary(mag), xyz.astype(np.float64), lam.astype(np.float64))
    sB, sG = abs_scales(mag, xyz, lam)
    assert (np.abs(got["B"].cpu().numpy() - B) <= TOL_FP64 * sB).all()
    assert (np.abs(got["gradB"].cpu().numpy() - G) <= TOL_FP64 * sG[:, :, None]).all()
    f.close()
