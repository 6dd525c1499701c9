"""Simplex steps whose warps hold one point, a few or 32, in one and in several passes over the
active list: a point's search does not depend on how many others run beside it.  FP64 form over
eight iterations on a 16 x 12 grid: the same decisions (iterations, evaluations, step codes), and
lambda to the rounding of sums whose partials are added in another order (1e-9)."""
import numpy as np
import pytest

from test_gpu_eval import random_mag, random_points

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("method", [0, 1])
def test_search_does_not_depend_on_company(mode, method):
    import paper_1306_1122_gb300 as dbie
    mag = random_mag(16, 12, 401)
    xyz, _ = random_points(mag, 40000, 402, zlo=0.4, zhi=9.0)
    f = dbie.DBIEField.from_magnetogram(mag)
    opt = dbie.Options(precision=1, lambda_mode=mode, method=method, max_iter=8)
    X = torch.from_numpy(xyz).cuda()
    full = f.solve(X, opt, codes=8)
    for part in (slice(0, 1), slice(7, 160), slice(1000, 6000)):
        r = f.solve(X[part], opt, codes=8)
        for k in ("iters", "nfev", "status", "codes"):
            assert torch.equal(r[k], full[k][part]), k
        assert torch.allclose(r["lam"], full["lam"][part], rtol=1e-9, atol=1e-12)
    f.close()
