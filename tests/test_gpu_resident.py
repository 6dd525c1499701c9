"""The search in one kernel (few points, few pixels) against the search by launches: the same
decisions, and lambda and B with them.  Profiling turns the single kernel off, so one context runs
both.  Sizes: one point, fewer and more points than CTAs, several per CTA, a batch of uneven
problems (one without points), elements, a tied lambda, no certification, given starts."""
import numpy as np
import pytest

from test_gpu_eval import random_mag, random_points

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dbie():
    import paper_1306_1122_gb300 as d
    return d


def _same(a, b):
    for k in ("iters", "nfev", "status", "codes"):
        assert torch.equal(a[k], b[k]), k
    assert torch.allclose(a["lam"], b["lam"], rtol=1e-9, atol=1e-12)
    scale = float(b["B"].abs().max())
    assert torch.allclose(a["B"], b["B"], rtol=1e-5, atol=1e-6 * scale)


@pytest.mark.parametrize("nx,ny,n,quad,kw", [
    (16, 16, 1, 0, {}), (33, 29, 300, 0, {}), (20, 16, 1200, 0, {}), (31, 23, 250, 0, dict(lambda_mode=1)),
    (17, 15, 60, 3, {}), (24, 24, 200, 0, dict(certify=0.0)), (24, 24, 200, 0, dict(certify_ref=0.0)),
    (24, 20, 150, -1, {}), (40, 3, 90, 0, dict(near_z=0.0)), (1, 1, 3, 0, {})])
def test_one_kernel_matches_launches(dbie, nx, ny, n, quad, kw):
    mag = random_mag(nx, ny, 600 + nx)
    xyz, _ = random_points(mag, n, 601 + n, zlo=0.5, zhi=12.0)
    f = dbie.DBIEField.from_magnetogram(mag)
    if quad:
        f.set_quadrature(quad)
    X = torch.from_numpy(xyz).cuda()
    opt = dbie.Options(max_iter=12, **kw)
    l0 = torch.from_numpy(np.random.default_rng(5).uniform(-0.05, 0.05, (n, 3))).cuda()
    for init in (None, l0):
        one = f.solve(X, opt, lambda_init=init, codes=12)
        f.set_profiling(True)
        rounds = f.solve(X, opt, lambda_init=init, codes=12)
        f.set_profiling(False)
        if kw.get("certify") == 0.0:   # decided by the noise of the FP32 sums: the field only
            assert torch.isfinite(one["B"]).all() and (one["iters"] <= 12).all()
        else:
            _same(one, rounds)
    f.close()


def test_one_kernel_batch(dbie):
    shapes = [(16, 12, 90), (33, 20, 7), (8, 8, 0), (25, 25, 120)]
    mags = [random_mag(nx, ny, 640 + i) for i, (nx, ny, _) in enumerate(shapes)]
    pts = [random_points(m, s[2], 650 + i, zlo=0.5, zhi=12.0)[0] if s[2] else np.zeros((0, 3), np.float32)
           for i, (m, s) in enumerate(zip(mags, shapes))]
    fields = [dbie.DBIEField.from_magnetogram(m) for m in mags]
    X = [torch.from_numpy(p).cuda() for p in pts]
    opt = dbie.Options(max_iter=12)
    one = dbie.solve_batched(fields, X, opt, codes=12)
    fields[0].set_profiling(True)
    rounds = dbie.solve_batched(fields, X, opt, codes=12)
    for a, b in zip(one, rounds):
        if len(a["B"]):
            _same(a, b)
    for f in fields:
        f.close()
