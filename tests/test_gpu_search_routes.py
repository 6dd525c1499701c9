"""The search in one kernel against the search by launches, which more points than the one kernel
takes bring about: a point's search does not depend on how many others run beside it.  The launches
that profiling counts say which of the two ran (one, or four rounds and more).  Without certification
the FP32 sums' rounding decides near ties, so only the field is compared, with FP64 at the returned
lambda (per term 1.5e-6 (1 + theta) + 4e-7 theta^2 of |b| / r^3, theta = lambda r, as derived in
test_gpu_half_turns.py; the near field is off there)."""
import numpy as np
import pytest

from test_gpu_eval import random_mag, random_points

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MORE = 1300


@pytest.fixture(scope="module")
def dbie():
    import paper_1306_1122_gb300 as d
    return d


def profiled(field, search, launches):
    field.set_profiling(True)
    field.stats(reset=True)
    r = search()
    st = field.stats(reset=True)
    field.set_profiling(False)
    assert launches(st["launches"]), st["launches"]
    assert st["objective_ms"] > 0 and st["kernel_ms"] >= st["objective_ms"] and st["objective_pairs"] > 0
    return r


def one(k):
    return k == 1


def many(k):
    return k >= 4


def same(a, b, n):
    for k in ("iters", "nfev", "status", "codes"):
        assert torch.equal(a[k], b[k][:n]), k
    assert torch.allclose(a["lam"], b["lam"][:n], rtol=1e-9, atol=1e-12)
    scale = float(b["B"].abs().max())
    assert torch.allclose(a["B"], b["B"][:n], rtol=1e-5, atol=1e-6 * scale)


@pytest.mark.parametrize("nx,ny,n,quad,kw", [
    (16, 16, 1, 0, {}), (33, 29, 300, 0, {}), (20, 16, 1200, 0, {}), (31, 23, 250, 0, dict(lambda_mode=1)),
    (17, 15, 60, 3, {}), (24, 24, 200, 0, dict(certify_ref=0.0)), (24, 20, 150, -1, {}),
    (40, 3, 90, 0, dict(near_z=0.0)), (1, 1, 3, 0, {}), (128, 128, 5, 0, {})])
def test_one_kernel_and_launches_agree(dbie, nx, ny, n, quad, kw):
    mag = random_mag(nx, ny, 700 + nx)
    xyz, _ = random_points(mag, n + MORE, 701 + n, zlo=0.5, zhi=12.0)
    f = dbie.DBIEField.from_magnetogram(mag)
    if quad:
        f.set_quadrature(quad)
    X = torch.from_numpy(xyz).cuda()
    opt = dbie.Options(max_iter=12, **kw)
    l0 = torch.from_numpy(np.random.default_rng(6).uniform(-0.05, 0.05, (n + MORE, 3))).cuda()
    for init in (None, l0):
        few = profiled(f, lambda: f.solve(X[:n], opt, lambda_init=None if init is None else init[:n],
                                          codes=12), one)
        plain = f.solve(X[:n], opt, lambda_init=None if init is None else init[:n], codes=12)
        all_ = profiled(f, lambda: f.solve(X, opt, lambda_init=init, codes=12), many)
        assert all(torch.equal(few[k], plain[k]) for k in ("iters", "nfev", "status", "codes"))
        same(few, all_, n)
    f.close()


def test_batch(dbie):
    shapes = [(16, 12, 90), (33, 20, 7), (8, 8, 0), (25, 25, 120)]
    mags = [random_mag(nx, ny, 740 + i) for i, (nx, ny, _) in enumerate(shapes)]
    fields = [dbie.DBIEField.from_magnetogram(m) for m in mags]
    X = [torch.from_numpy(random_points(m, s[2] + MORE, 750 + i, zlo=0.5, zhi=12.0)[0]).cuda()
         for i, (m, s) in enumerate(zip(mags, shapes))]
    opt = dbie.Options(max_iter=12)
    few = profiled(fields[0], lambda: dbie.solve_batched(fields, [x[:s[2]] for x, s in zip(X, shapes)],
                                                         opt, codes=12), one)
    all_ = profiled(fields[0], lambda: dbie.solve_batched(fields, X, opt, codes=12), many)
    for a, b, s in zip(few, all_, shapes):
        if s[2]:
            same(a, b, s[2])
    for f in fields:
        f.close()


@pytest.mark.parametrize("n", [200, 200 + MORE])
def test_field_without_certification(dbie, n):
    mag = random_mag(24, 24, 760)
    xyz, _ = random_points(mag, n, 761, zlo=0.5, zhi=12.0)
    f = dbie.DBIEField.from_magnetogram(mag)
    X = torch.from_numpy(xyz).cuda()
    r = profiled(f, lambda: f.solve(X, dbie.Options(max_iter=12, certify=0.0, near_z=0.0)),
                 one if n <= 200 else many)
    f.close()
    j, i = np.mgrid[0:24, 0:24].astype(np.float64)
    P, lam = xyz.astype(np.float64), r["lam"].cpu().numpy()
    d = np.sqrt((P[:, :1] - (mag.x0 + i * mag.hx).ravel()) ** 2 +
                (P[:, 1:2] - (mag.y0 + j * mag.hy).ravel()) ** 2 + P[:, 2:] ** 2)
    for p, b in enumerate((mag.Bx, mag.By, mag.Bz)):
        b = np.asarray(b, np.float64).ravel()
        th = lam[:, p:p + 1] * d
        w = P[:, 2:] / d ** 3 * (mag.dA / (2 * np.pi))
        err = w * (1.5e-6 * (1 + th) + 4e-7 * th ** 2) @ abs(b)
        assert (abs(r["B"][:, p].cpu().numpy() - w * (th * np.sin(th) + np.cos(th)) @ b) <= err).all()


@pytest.mark.parametrize("nx,ny,n,route", [(128, 128, 4, one), (129, 128, 1, many), (150, 131, 3, many),
                                           (256, 256, 2, many)])
def test_few_points_over_many_pixels(dbie, nx, ny, n, route):
    """Past 128 strips of 128 pixels even one point's search goes by launches; the decisions are the
    FP64 form's, and B is certified to 1e-5."""
    mag = random_mag(nx, ny, 770 + nx)
    xyz, _ = random_points(mag, n, 771, zlo=0.5, zhi=12.0)
    f = dbie.DBIEField.from_magnetogram(mag)
    X = torch.from_numpy(xyz).cuda()
    r = profiled(f, lambda: f.solve(X, dbie.Options(max_iter=12), codes=12), route)
    d = f.solve(X, dbie.Options(max_iter=12, precision=1), codes=12)
    f.close()
    for k in ("iters", "nfev", "status", "codes"):
        assert torch.equal(r[k], d[k]), k
    assert torch.allclose(r["lam"], d["lam"], rtol=1e-9, atol=1e-12)
    assert ((r["B"] - d["B"]).norm(dim=1) <= 1e-5 * d["B"].norm(dim=1)).all()
