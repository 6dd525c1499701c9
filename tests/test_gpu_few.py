"""The kernel for few queries (the lanes of a warp take pixels) at the edges of its strips (128
pixels), tiles, ranges and warps, on both sides of its dispatch rule, against the FP64 oracle with
the mixed form's gates (gates.py); and searches on both sides of the rule, which must take the same
decisions."""
import numpy as np
import pytest

import oracle
from gates import abs_scales, check_B, check_grad, oracle_boundary
from test_gpu_eval import random_mag, random_points, run_eval

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dbie():
    import paper_1306_1122_gb300 as d
    return d


@pytest.mark.parametrize("nx,ny,n", [(1, 1, 1), (16, 8, 3), (129, 1, 40), (16, 16, 129),
                                     (257, 3, 2), (40, 33, 2500), (40, 33, 2501), (30, 20, 6000),
                                     (30, 20, 6001), (300, 251, 7)])
def test_sums_at_sizes(dbie, nx, ny, n):
    mag = random_mag(nx, ny, 500 + nx, x0=-2.0, y0=1.0)
    xyz, lam = random_points(mag, n, 501 + n, zlo=0.4, zhi=25.0)
    bd = oracle_boundary(mag)
    B, G, dl = oracle.field(bd, xyz.astype(np.float64), lam.astype(np.float64))
    sB, sG = abs_scales(mag, xyz, lam)
    f = dbie.DBIEField.from_magnetogram(mag)
    X, L = torch.from_numpy(xyz), torch.from_numpy(lam)
    value = f.eval(X, L)["B"].cpu().numpy()
    vl = {k: v.cpu().numpy() for k, v in f.eval(X, L, dlam=True).items()}
    obj = {k: v.cpu().numpy() for k, v in f.objective(X, L).items()}
    f.close()
    full = run_eval(dbie, mag, xyz, lam, 0)   # B, gradient, dB/dlambda, f, g
    for got in (value, vl["B"], full["B"]):
        assert check_B(got, B, sB)["bad"].size == 0
    assert check_grad(full["gradB"], G, sG[:, :, None])["ok"]
    for got in (vl["dBdlam"], full["dBdlam"]):
        assert check_grad(got, dl, np.abs(dl).max() + 1e-30)["ok"]
    # the gradient variant's sums are the objective's: f, g of both calls agree to FP32 terms
    for k in ("f", "g"):
        assert np.allclose(obj[k], full[k], rtol=2e-3, atol=2e-4), k


def test_elements_few(dbie):
    mag = random_mag(31, 23, 520)
    xyz, lam = random_points(mag, 65, 521, zlo=0.6, zhi=12.0)
    bd = oracle_boundary(mag)
    B, G, _ = oracle.field(bd, xyz.astype(np.float64), lam.astype(np.float64), quad_order=3)
    f = dbie.DBIEField.from_magnetogram(mag)
    f.set_quadrature(3)
    r = f.eval(torch.from_numpy(xyz), torch.from_numpy(lam), grad=True)
    sB, sG = abs_scales(mag, xyz, lam)
    assert check_B(r["B"].cpu().numpy(), B, sB)["bad"].size == 0
    assert check_grad(r["gradB"].cpu().numpy(), G, sG[:, :, None])["ok"]
    f.close()


@pytest.mark.parametrize("mode", [0, 1])
def test_search_same_on_both_sides_of_the_rule(dbie, mode):
    mag = random_mag(24, 20, 530)
    xyz, _ = random_points(mag, 13000, 531, zlo=0.5, zhi=15.0)
    f = dbie.DBIEField.from_magnetogram(mag)
    X = torch.from_numpy(xyz).cuda()
    opt = dbie.Options(lambda_mode=mode, max_iter=10)
    dense = f.solve(X, opt, codes=10)                # above the rule's 12,000 points
    for part in (slice(0, 1), slice(100, 800), slice(1000, 13000)):
        few = f.solve(X[part], opt, codes=10)
        for k in ("iters", "nfev", "status", "codes"):
            assert torch.equal(few[k], dense[k][part]), k
        assert torch.allclose(few["lam"], dense["lam"][part], rtol=1e-9, atol=1e-12)
        scale = dense["B"].abs().max()
        assert torch.allclose(few["B"], dense["B"][part], rtol=1e-5, atol=1e-6 * float(scale))
    f.close()
