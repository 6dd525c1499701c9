"""A certified search that starts at lambdas where the FP32 error bounds leave FP32's range: the bound
of such a value certifies nothing, so every comparison it takes part in counts as a near tie and is
re-evaluated (at least the sort of the first vertices, for every point), by launches and in the one
kernel alike; the decisions are those of a band so wide that every comparison ties."""
import numpy as np
import pytest

from test_gpu_eval import random_mag, random_points

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lam0", [1e13, 1e16])
@pytest.mark.parametrize("mode,n", [(0, 40), (1, 40), (0, 1300)])
def test_bound_beyond_range_is_a_tie(lam0, mode, n):
    import paper_1306_1122_gb300 as dbie
    mag = random_mag(16, 12, 31)
    xyz, _ = random_points(mag, n, 32, zlo=0.5, zhi=9.0)
    f = dbie.DBIEField.from_magnetogram(mag)
    X = torch.from_numpy(xyz).cuda()
    l0 = torch.from_numpy(lam0 * np.random.default_rng(33).uniform(0.5, 1.0, (n, 3))).cuda()
    runs = []
    for kw in ({}, dict(certify=1e6, certify_ref=0.0)):
        f.stats(reset=True)
        runs.append(f.solve(X, dbie.Options(max_iter=2, lambda_mode=mode, simplex_step=0.3 * lam0, **kw),
                            lambda_init=l0, codes=2))
        assert f.stats()["ties"] >= n
    for k in ("iters", "nfev", "status", "codes"):
        assert torch.equal(runs[0][k], runs[1][k]), k
    f.close()
