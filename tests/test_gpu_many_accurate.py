"""Accurate sums of many points over few pixels, one query per thread, against the same points in a
call of few (one query per CTA and pixel range) and against the FP64 form: differences within the
two calls' own worst-case bounds (which agree to 1e-4, the accuracy they are summed to), float-float
sums within the gate of test_gpu_ff.py, 1e-11, of the terms' absolute-value sums (u = theta sin + cos
taken as 1 + theta), and 6e-14 of the largest angle more (theta's own 2^-45, twice).  Sizes at and past
the rule's edges, blocks with a remainder, several tiles and one, elements, a tied lambda, and angles
beyond the table's reduction."""
import numpy as np
import pytest

from test_gpu_eval import random_mag, random_points
from test_gpu_ff import TOL_FF

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _setup(nx, ny, n, quad, seed, lmax=0.3):
    import paper_1306_1122_gb300 as dbie
    mag = random_mag(nx, ny, seed)
    xyz, lam = random_points(mag, n, seed + 1, zlo=0.4, zhi=12.0, lam=lmax)
    f = dbie.DBIEField.from_magnetogram(mag)
    if quad:
        f.set_quadrature(quad)
    return dbie, mag, f, torch.from_numpy(xyz).cuda(), torch.from_numpy(lam).cuda()


@pytest.mark.parametrize("nx,ny,n,quad,tied", [
    (1, 1, 12000, 0, False), (16, 16, 12001, 0, False), (40, 33, 12127, 0, False), (17, 15, 13000, 3, False),
    (16, 17, 6000, 0, True), (30, 30, 6333, 0, True), (24, 20, 12500, -1, False)])
def test_differences(nx, ny, n, quad, tied):
    dbie, _, f, X, lam = _setup(nx, ny, n, quad, 820 + nx)
    l0 = lam.double()
    l1 = l0 + 0.02 * torch.rand(n, 3, dtype=torch.float64, device="cuda",
                                generator=torch.Generator("cuda").manual_seed(5))
    S, E = f.eval_difference(X, l1, l0, tied=tied)
    part = torch.cat([torch.arange(0, 200), torch.arange(n - 200, n)]).cuda()
    s, e = f.eval_difference(X[part], l1[part], l0[part], tied=tied)
    f.close()
    assert torch.allclose(E[part], e, rtol=1e-4, atol=0.0)
    assert ((S[part] - s).abs() <= E[part] + e).all()


@pytest.mark.parametrize("nx,ny,n,quad,lmax", [
    (1, 1, 150000, 0, 0.3), (16, 16, 150001, 0, 0.3), (16, 16, 150100, 0, 2000.0), (25, 24, 300050, 0, 0.3),
    (9, 9, 160000, 3, 0.3)])
def test_float_float(nx, ny, n, quad, lmax):
    dbie, mag, f, X, lam = _setup(nx, ny, n, quad, 850 + nx, lmax)
    got = f.eval(X, lam, grad=True, options=dbie.Options(precision=2))
    val = f.eval(X, lam, options=dbie.Options(precision=2))["B"]
    part = torch.cat([torch.arange(0, 300), torch.arange(n - 300, n)]).cuda()
    ref = f.eval(X[part], lam[part], grad=True, options=dbie.Options(precision=1))
    few = f.eval(X[part], lam[part], grad=True, options=dbie.Options(precision=2))
    f.close()
    if quad:   # (no absolute-value sums of elements here: the call of few points within its own accuracy)
        scale = few["B"].abs().max()
        assert ((got["B"][part] - few["B"]).abs() <= 1e-10 * scale).all()
        return
    j, i = np.mgrid[0:ny, 0:nx].astype(np.float64)
    P, L = X[part].cpu().numpy().astype(np.float64), abs(lam[part].cpu().numpy().astype(np.float64))
    dx, dy = abs(P[:, :1] - (mag.x0 + i * mag.hx).ravel()), abs(P[:, 1:2] - (mag.y0 + j * mag.hy).ravel())
    r = np.sqrt(dx ** 2 + dy ** 2 + P[:, 2:] ** 2)
    tol = TOL_FF + 6e-14 * float((L.max(1, keepdims=True) * r).max())
    for p, b in enumerate((mag.Bx, mag.By, mag.Bz)):
        b = abs(np.asarray(b, np.float64)).ravel() * mag.dA / (2 * np.pi)
        u = (1 + L[:, p:p + 1] * r) / r ** 3
        w = P[:, 2:] * (L[:, p:p + 1] ** 2 / r ** 3 + 3 * u / r ** 2)
        sB, sG = P[:, 2] * (u @ b), (u + w * (dx + dy + P[:, 2:])) @ b
        want = ref["B"][:, p].cpu().numpy()
        for out in (got["B"][part], val[part]):
            assert (abs(out[:, p].cpu().numpy() - want) <= tol * sB).all()
        err = (got["gradB"][part] - ref["gradB"])[:, p].abs().amax(1).cpu().numpy()
        assert (err <= tol * sG).all()
