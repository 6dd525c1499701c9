"""dL/dlambda of the adjoint from the cosine sums alone, against gB dB/dlambda of an evaluation (which
computes them beside the field with the same FP32 terms: 2e-6 of the largest value; FP64 form:
1e-12), on both sides of the rule for few queries, at points in and above the near field."""
import numpy as np
import pytest

from test_gpu_eval import random_mag, random_points

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,n,quad,prec", [
    (1, 1, 1, 0, 0), (33, 17, 40, 0, 0), (36, 20, 2500, 0, 0), (36, 20, 7000, 0, 0), (35, 21, 7000, 0, 0),
    (15, 13, 50, 2, 0), (15, 13, 7000, 2, 0), (20, 16, 60, -1, 0), (20, 16, 60, 0, 1)])
def test_lambda_gradient(nx, ny, n, quad, prec):
    import paper_1306_1122_gb300 as dbie
    mag = random_mag(nx, ny, 700 + nx)
    xyz, lam = random_points(mag, n, 701 + n, zlo=0.5, zhi=9.0)
    f = dbie.DBIEField.from_magnetogram(mag)
    if quad:
        f.set_quadrature(quad)
    opt = dbie.Options(precision=prec)
    gB = torch.from_numpy(np.random.default_rng(7).normal(size=(n, 3))).cuda()
    X, L = torch.from_numpy(xyz).cuda(), torch.from_numpy(lam).cuda()
    want = gB * f.eval(X, L, dlam=True, options=opt)["dBdlam"]
    got = f.vjp(X, L.double(), gB, options=opt)[1]
    tol = 1e-12 if prec else 2e-6
    assert float((got - want).abs().max()) <= tol * float(want.abs().max())
    f.close()
