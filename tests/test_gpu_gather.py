"""Sums of many splits, gathered by the warps of a CTA, against the same points and pixels in calls
of few splits (a thread each): FP64 form, so both sides differ by the order of the partial sums
alone (1,800 terms: 1e-12 of the largest value; f, g and their gradients, quotients of sums that
cancel, 1e-8)."""
import numpy as np
import pytest

from test_gpu_eval import random_mag, random_points

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 33, 300, 8192, 9000])
def test_gathered_splits(n):
    import paper_1306_1122_gb300 as dbie
    mag = random_mag(45, 40, 60)
    xyz, lam = random_points(mag, 70000, 61, zlo=0.5, zhi=9.0)
    f = dbie.DBIEField.from_magnetogram(mag)
    opt = dbie.Options(precision=1)
    X, L = torch.from_numpy(xyz).cuda(), torch.from_numpy(lam).cuda()
    kw = dict(grad=True, dlam=True, objective=True, options=opt)
    a, b = f.eval(X[:n], L[:n], **kw), f.eval(X, L, **kw)
    a.update(f.objective(X[:n], L[:n], opt))
    b.update(f.objective(X, L, opt))
    for k in a:
        tol = 1e-12 if k in ("B", "gradB", "dBdlam") else 1e-8
        want = b[k][:n]
        assert float((a[k] - want).abs().max()) <= tol * float(b[k].abs().max()), k
    gB = torch.from_numpy(np.random.default_rng(5).normal(size=(n, 3))).cuda()
    got = f.vjp(X[:n], L[:n].double(), gB, glam=False, options=opt)[0]
    want = torch.zeros_like(got)
    for i in range(0, n, 1000):
        k = slice(i, min(n, i + 1000))
        f.vjp(X[k], L[k].double(), gB[k], glam=False, options=opt, gB0=want)
    assert float((got - want).abs().max()) <= 1e-12 * float(want.abs().max())
    f.close()
