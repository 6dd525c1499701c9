"""Lambdas that are infinite, NaN or far beyond any angle's resolution, at fixed lambda.  B and its
lambda-derivative of a component whose lambda is infinite or NaN are NaN, in every component alike
(one of them takes its sine and cosine from polynomials); a finite lambda, however large, gives finite
sums, and up to angles of 1.5e10 rad sums of bounded sines and cosines: |B_p| <=
z sum (|lambda_p| r + 1) |b| / r^3, with 0.1 % for rounding.
On both sides of the rule for few points, on rows of four and others, with and without the near field."""
import numpy as np
import pytest

from test_gpu_eval import random_mag, random_points

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,n", [(20, 13, 30), (19, 14, 30), (20, 13, 7000), (19, 14, 7000)])
@pytest.mark.parametrize("near", [0.0, 2.0])
def test_lambda_out_of_range(nx, ny, n, near):
    import paper_1306_1122_gb300 as dbie
    mag = random_mag(nx, ny, 70 + nx)
    xyz, _ = random_points(mag, n, 71 + n, zlo=0.4, zhi=20.0)
    vals = torch.tensor([0.1, -0.2, float("inf"), float("-inf"), float("nan"), -3e12, 1e8, 1e20]).cuda()
    lam = vals[torch.arange(3 * n, device="cuda").reshape(n, 3) * 5 % 7 * 3 % 8]
    lam = torch.where(torch.arange(n, device="cuda")[:, None] % 5 == 0, vals[2], lam)
    X, bad = torch.from_numpy(xyz).cuda(), ~torch.isfinite(lam)
    gB = torch.ones(n, 3, dtype=torch.float64, device="cuda")
    f = dbie.DBIEField.from_magnetogram(mag)
    opt = dbie.Options(near_z=near)
    r = f.eval(X, lam, dlam=True, options=opt)
    B = f.eval(X, lam, options=opt)["B"]
    glam = f.vjp(X, lam.double(), gB, options=opt)[1]
    f.close()
    for out in (B, r["B"], r["dBdlam"], glam):
        assert torch.isnan(out[bad]).all() and torch.isfinite(out[~bad]).all()
    j, i = np.mgrid[0:ny, 0:nx].astype(np.float64)
    P = xyz.astype(np.float64)
    d = np.sqrt((P[:, :1] - (mag.x0 + i * mag.hx).ravel()) ** 2 +
                (P[:, 1:2] - (mag.y0 + j * mag.hy).ravel()) ** 2 + P[:, 2:] ** 2)
    lc = abs(lam.double().cpu().numpy())
    known = lc <= 1e8
    lc[~known] = 0.0
    for p, b in enumerate((mag.Bx, mag.By, mag.Bz)):
        most = 1.001 * P[:, 2] * ((lc[:, p:p + 1] * d + 1) / d ** 3 * (mag.dA / (2 * np.pi)) @
                                  abs(np.asarray(b, np.float64)).ravel())
        for out in (B, r["B"]):
            o = out[:, p].cpu().numpy()
            assert (abs(o) <= most)[known[:, p]].all()
