"""FP32 sums whose sine and cosine of one component are polynomials on the FMA pipe: B (with and
without dB/dlambda) and the adjoint against FP64, for lambda r up to ~600 and on both sides of the
rules for few points and for rows of four.  The bound is the sum of the terms' own errors.  With
theta = lambda r and phi = (theta sin + cos) / r^3: sine, cosine 5e-7, four roundings and 1 / r^3
(3 x 1.2e-7) make 1.1e-6 (1 + theta), taken as 1.5e-6; theta is off by 3.4e-7 of itself (1 / r,
two products, 1 / 2 pi), taken as 4e-7 theta^2."""
import numpy as np
import pytest

from test_gpu_eval import random_mag, random_points

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,n", [(1, 1, 1), (20, 13, 40), (19, 14, 301), (20, 13, 13000), (19, 14, 13000)])
@pytest.mark.parametrize("lmax", [0.0, 0.3, 20.0])
def test_half_turn_sums(nx, ny, n, lmax):
    import paper_1306_1122_gb300 as dbie
    mag = random_mag(nx, ny, 50 + nx)
    xyz, _ = random_points(mag, n, 51 + n, zlo=0.4, zhi=20.0)
    rng = np.random.default_rng(52)
    lam = (lmax * rng.uniform(-1, 1, (n, 3))).astype(np.float32)
    gB = rng.normal(size=(n, 3))
    f = dbie.DBIEField.from_magnetogram(mag)
    X, L = torch.from_numpy(xyz).cuda(), torch.from_numpy(lam).cuda()
    opt = dbie.Options(near_z=0.0)
    B = f.eval(X, L, options=opt)["B"].cpu().numpy()
    B2 = f.eval(X, L, dlam=True, options=opt)["B"].cpu().numpy()
    gB0 = f.vjp(X, L.double(), torch.from_numpy(gB).cuda(), glam=False, options=opt)[0].cpu().numpy()
    f.close()
    j, i = np.mgrid[0:ny, 0:nx].astype(np.float64)
    P = xyz.astype(np.float64)
    xk, yk = (mag.x0 + i * mag.hx).ravel(), (mag.y0 + j * mag.hy).ravel()
    r = np.sqrt((P[:, :1] - xk) ** 2 + (P[:, 1:2] - yk) ** 2 + P[:, 2:] ** 2)
    for p, b in enumerate((mag.Bx, mag.By, mag.Bz)):
        th = lam[:, p:p + 1].astype(np.float64) * r
        phi = P[:, 2:] * (th * np.sin(th) + np.cos(th)) / r ** 3 * (mag.dA / (2 * np.pi))
        err = P[:, 2:] / r ** 3 * (mag.dA / (2 * np.pi)) * (1.5e-6 * (1 + abs(th)) + 4e-7 * th ** 2)
        b = np.asarray(b, np.float64).ravel()
        assert (abs(B[:, p] - phi @ b) <= err @ abs(b)).all()
        assert (abs(B2[:, p] - phi @ b) <= err @ abs(b)).all()
        g = gB0.reshape(-1, 3)[:, p]
        assert (abs(g - phi.T @ gB[:, p]) <= err.T @ abs(gB[:, p])).all()
