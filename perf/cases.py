"""Workloads of the DBIE library for timing: what its users have it do, through its public calls.

A case is a dict of plain values:

  kind       "eval"    DBIEField.eval at fixed lambda (Eq. 16)
             "train"   dbie_apply forward and backward (gradients of B0 and lambda)
             "search"  dbie_solve_apply forward and backward (gradient through the lambda search)
             "solve"   DBIEField.solve, the per-point lambda search
             "batch"   solve_batched over several magnetograms
  nx, ny     magnetogram size in pixels ("batch": the largest; the sides are drawn between 32 and it)
  h          pixel spacing (the length unit is the caller's: pixels, or Mm)
  n          evaluation points ("batch": the most of one problem)
  layout     "grid": points above pixel centres, layer by layer; "scatter": anywhere in the field of view
  form       "mixed", "float_float" or "fp64"
  grad       eval: also grad B, f and g
  quad       0: pixel centres; 1..8: nine-node elements; -1: exact near field
  tied       one lambda per point instead of one per component
  max_iter   simplex iterations of the search

The magnetograms are sheared active regions with noise (the recipe of the repository's synthetic
workloads), the points lie 0.5 to 48 pixels above them, and the fixed lambdas follow the
distribution that the search returns on such regions (median 0.03 per pixel, a quarter near 0,
tails to 0.3).

The mixed form is single-precision arithmetic (FP32 pair terms; B to 1e-5), so programs carry its
fields on in float32, the type of the points and the magnetogram, and so do these cases.  The
float-float and FP64 forms are called for more, and keep float64; so does the searched lambda,
which the certified search determines to FP64's decisions.
"""
import math

import torch

import paper_1306_1122_gb300 as dbie

FORMS = {"mixed": 0, "fp64": 1, "float_float": 2}


def _case(kind, nx, ny, n, **more):
    c = dict(kind=kind, nx=nx, ny=ny, h=1.0, n=n, layout="scatter", form="mixed", grad=False,
             quad=0, tied=False, max_iter=50)
    c.update(more)
    return c


def listed():
    cases = dict(
        # one step of a field-line tracer: the field at the heads of some lines
        trace_step=_case("eval", 128, 128, 64),
        # a probe of a small ragged cut-out, with the force-free and divergence measures
        eval_ragged=_case("eval", 129, 70, 300, grad=True, h=0.72),
        # a slab of a coronal volume above a large region
        eval_slab=_case("eval", 512, 256, 49152, layout="grid"),
        # field, gradient and f, g at scattered points: the quality map of a finished model
        eval_quality=_case("eval", 300, 300, 20000, grad=True, h=0.72),
        # the nine-node element rule of Eq. 15
        eval_elements=_case("eval", 129, 129, 4096, grad=True, quad=3),
        # accurate fields: float-float, and the plain FP64 form that others are checked against
        eval_float_float=_case("eval", 128, 128, 4096, grad=True, form="float_float"),
        eval_fp64=_case("eval", 64, 64, 2048, form="fp64"),
        # fitting a magnetogram and lambda to observed fields: one forward and backward pass
        train_fixed=_case("train", 128, 128, 32768, layout="grid"),
        # the same through the lambda search
        train_search=_case("search", 64, 64, 1024),
        # the search on a small box, to convergence
        solve_small=_case("solve", 32, 32, 2048, layout="grid"),
        # ten search iterations over a volume
        solve_volume=_case("solve", 128, 128, 131072, layout="grid", max_iter=10),
        # many magnetograms of uneven size in one call, to convergence
        solve_batch=_case("batch", 128, 128, 300, nprob=16),
    )
    return [dict(c, name=name) for name, c in cases.items()]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "train", "search", "solve", "solve", "batch"])
    c = _case(kind, 0, 0, 0, h=rng.choice([1.0, 1.0, 0.72, 2.0]),
              layout=rng.choice(["grid", "scatter"]))
    if kind == "eval":
        c["form"] = rng.choice(["mixed", "mixed", "mixed", "float_float", "fp64"])
        c["grad"] = rng.random() < 0.5
        c["quad"] = rng.choice([0, 0, 0, -1, 2, 4])
        c["nx"], c["ny"] = _log(rng, 17, 512), _log(rng, 17, 300)
        if c["quad"] > 0:   # elements need odd sides
            c["nx"], c["ny"] = _log(rng, 17, 160) | 1, _log(rng, 17, 160) | 1
        c["grad"] &= c["quad"] >= 0
        most = {"mixed": 6e9, "float_float": 2e8, "fp64": 2e7}[c["form"]]
        c["n"] = _log(rng, 16, max(32, min(50000, most / (c["nx"] * c["ny"] * max(1, c["quad"]) ** 2))))
    elif kind == "train":
        c["nx"], c["ny"] = _log(rng, 24, 256), _log(rng, 24, 256)
        c["n"] = _log(rng, 100, 32768)
    elif kind == "search":
        c["nx"], c["ny"] = _log(rng, 24, 128), _log(rng, 24, 128)
        c["n"] = _log(rng, 50, 1500)
    elif kind == "solve":
        c["nx"], c["ny"] = _log(rng, 24, 256), _log(rng, 24, 256)
        c["tied"] = rng.random() < 0.25
        if rng.random() < 0.5:
            c["n"] = _log(rng, 50, 2500)
        else:
            c["max_iter"], c["n"] = 10, _log(rng, 1000, 50000)
    else:
        c["nx"] = c["ny"] = _log(rng, 48, 160)
        c["nprob"], c["n"] = rng.randint(4, 24), _log(rng, 50, 250)
    return c


# ------------------------------------------------------------------------------ inputs ----
def _region(nx, ny, h, g):
    """Bx, By, Bz (ny, nx) float32 of a sheared active region of four flux patches plus noise."""
    u = torch.rand(4, 4, generator=g, dtype=torch.float64, device="cuda").tolist()
    y, x = torch.meshgrid(torch.arange(ny, device="cuda", dtype=torch.float64),
                          torch.arange(nx, device="cuda", dtype=torch.float64), indexing="ij")
    Bz, gx, gy = (torch.zeros(ny, nx, device="cuda", dtype=torch.float64) for _ in range(3))
    for q, (a, b, c, d) in enumerate(u):
        cx, cy = (0.2 + 0.6 * a) * nx, (0.2 + 0.6 * b) * ny
        s = max(2.0, (0.05 + 0.06 * c) * min(nx, ny))
        e = (500 + 1500 * d) * (-1) ** q * torch.exp(-((x - cx) ** 2 + (y - cy) ** 2) / (2 * s * s))
        Bz += e
        gx -= (x - cx) / s ** 2 * e
        gy -= (y - cy) / s ** 2 * e
    B = torch.stack([-5 * gx - 10 * gy, -5 * gy + 10 * gx, Bz])
    return (B + 10 * torch.randn(B.shape, generator=g, dtype=torch.float64, device="cuda")).float()


def _points(c, nx, ny, n, g):
    """(n, 3) float32 points above the field of view."""
    if c["layout"] == "grid":   # above pixel centres of the central part, layer by layer
        layers = min(32, max(1, n // 64))
        m = math.ceil(math.sqrt(n / layers))
        mx, my = min(m, nx), min(m, ny)
        k = torch.arange(n, device="cuda")
        x = (nx - mx) // 2 + k % mx
        y = (ny - my) // 2 + k // mx % my
        p = torch.stack([x.double(), y.double(), 1.0 + (k // (mx * my)).double()], 1)
    else:
        u = torch.rand(n, 3, generator=g, dtype=torch.float64, device="cuda")
        p = u * torch.tensor([nx - 1.0, ny - 1.0, 47.5], device="cuda", dtype=torch.float64)
        p[:, 2] += 0.5
    return (p * c["h"]).float()


def _lambdas(c, n, g):
    lam = 0.06 * torch.randn(n, 3, generator=g, dtype=torch.float64, device="cuda")
    u = torch.rand(n, 3, generator=g, dtype=torch.float64, device="cuda")
    lam = torch.where(u < 0.25, 0.02 * lam, torch.where(u > 0.995, 2.0 * lam, lam))
    return (lam / c["h"]).float()


def _inputs(c, seed):
    """(B0, points, lambda, upstream gradient) per problem, from the seed alone."""
    g = torch.Generator("cuda")
    g.manual_seed(seed)
    sizes = [(c["nx"], c["ny"], c["n"])]
    if c["kind"] == "batch":   # the sides and point counts belong to the case, not to the seed
        s = torch.Generator()
        s.manual_seed(c["nx"] * 1000003 + c["n"] * 1009 + c["nprob"])
        r = torch.rand(c["nprob"], 3, generator=s, dtype=torch.float64).tolist()
        side = lambda u: 32 + int(u * (c["nx"] - 31))
        sizes = [(side(a), side(b), max(16, int(d * c["n"]))) for a, b, d in r]
    return [(_region(nx, ny, c["h"], g), _points(c, nx, ny, n, g), _lambdas(c, n, g),
             torch.randn(n, 3, generator=g, device="cuda")) for nx, ny, n in sizes]


def prepare(case, seed):
    sets = _inputs(case, seed)
    fields = [dbie.DBIEField(*B, hx=case["h"], hy=case["h"]) for B, _, _, _ in sets]
    if case["quad"]:
        fields[0].set_quadrature(case["quad"])
    opt = dbie.Options(precision=FORMS[case["form"]], lambda_mode=int(case["tied"]),
                       max_iter=case["max_iter"])
    B, xyz, lam, up = sets[0]
    s = dict(case=case, fields=fields, points=[p for _, p, _, _ in sets], options=opt, xyz=xyz,
             lam=lam, up=up)
    if case["kind"] in ("train", "search"):   # B0 as (ny, nx, 3), the layout of the autograd calls
        s["B0"] = B.permute(1, 2, 0).contiguous().requires_grad_()
        s["lam"] = lam.requires_grad_()
    return s


# --------------------------------------------------------------------------------- run ----
def _kept(r):
    """A search's results as a program keeps them: single-precision fields, the searched lambda."""
    return {k: v.float() if k in ("B", "f", "g") else v for k, v in r.items()}


def run(s):
    c, field = s["case"], s["fields"][0]
    if c["kind"] == "eval":
        r = field.eval(s["xyz"], s["lam"], grad=c["grad"], objective=c["grad"], options=s["options"])
        return {k: v.float() for k, v in r.items()} if c["form"] == "mixed" else r
    if c["kind"] == "train":
        B = dbie.dbie_apply(field, s["B0"], s["lam"], s["xyz"], s["options"]).float()
        gB0, glam = torch.autograd.grad(B, (s["B0"], s["lam"]), s["up"])
        return {"B": B.detach(), "gB0": gB0, "glam": glam}
    if c["kind"] == "search":
        B, lam = dbie.dbie_solve_apply(field, s["B0"], s["xyz"], s["options"])
        B = B.float()
        gB0, = torch.autograd.grad(B, s["B0"], s["up"])
        return {"B": B.detach(), "lam": lam, "gB0": gB0}
    if c["kind"] == "solve":
        return _kept(field.solve(s["xyz"], s["options"]))
    rs = [_kept(r) for r in dbie.solve_batched(s["fields"], s["points"], s["options"])]
    return {k: torch.cat([r[k] for r in rs]) for k in rs[0]}


def work(case):
    """Bytes: inputs once, outputs once.  Operations per point and quadrature point: the distance
    and three sines, cosines and products of Eq. 16, and the derivative terms where asked for."""
    sizes = [(p.shape[0], B[0].numel()) for B, p, _, _ in _inputs(case, 0)]
    n, npix = sum(a for a, _ in sizes), sum(b for _, b in sizes)
    pairs = sum(a * b for a, b in sizes) * (0.25 * case["quad"] ** 2 if case["quad"] > 0 else 1)
    value, objective = 8 + 3 * 6, 8 + 3 * 13
    if case["kind"] == "eval":
        out = (15 if case["grad"] else 3) * (4 if case["form"] == "mixed" else 8)
        return {"bytes": 12 * npix + n * (24 + out),
                "flops": pairs * (objective if case["grad"] else value)}
    if case["kind"] == "train":   # the value, its lambda-derivative and the adjoint
        return {"bytes": 12 * npix * 2 + n * 60, "flops": pairs * (value + 6 + value)}
    # evaluations per point: four to begin with, and about 1.7 an iteration
    evals = 4 + 1.7 * min(48, case["max_iter"])
    flops = pairs * evals * objective
    if case["kind"] == "search":
        flops += pairs * 2 * objective
    return {"bytes": 12 * npix + n * (12 + 56), "flops": flops}


# ------------------------------------------------------------------------------- exact ----
def _gauss(m):
    """Gauss-Legendre abscissae and weights on [-1, 1] from the symmetric tridiagonal (Golub and
    Welsch)."""
    k = torch.arange(1, m, dtype=torch.float64)
    b = k / torch.sqrt(4 * k * k - 1)
    x, v = torch.linalg.eigh(torch.diag(b, 1) + torch.diag(b, -1))
    return x, 2 * v[0] ** 2


def _quadrature(c, B):
    """Positions (N, 2) of the quadrature points and b (3, N) = B0 times their weight / 2 pi."""
    h, (ny, nx) = c["h"], B.shape[1:]
    B = B.double()
    if c["quad"] > 0:   # biquadratic interpolation to the Gauss points of 2 x 2-interval elements
        x, w = _gauss(c["quad"])
        shape = torch.stack([x * (x - 1) / 2, 1 - x * x, x * (x + 1) / 2])   # node, Gauss point

        def axis(nodes):
            el = (nodes - 1) // 2
            at = (2 * torch.arange(el)[:, None] + 1 + x[None]).reshape(-1) * h
            M = torch.zeros(el, len(x), nodes, dtype=torch.float64)
            for e in range(el):
                M[e, :, 2 * e:2 * e + 3] = shape.T * w[:, None] * h
            return at.cuda(), M.reshape(-1, nodes).cuda()
        X, Mx = axis(nx)
        Y, My = axis(ny)
        b = My @ B @ Mx.T
    else:
        X, Y = (torch.arange(m, device="cuda", dtype=torch.float64) * h for m in (nx, ny))
        b = B * (h * h)
    yy, xx = torch.meshgrid(Y, X, indexing="ij")
    return torch.stack([xx.reshape(-1), yy.reshape(-1)], 1), b.reshape(3, -1) / (2 * math.pi)


def _chunks(n, N):
    step = max(1, int(3e7) // N)
    return [slice(i, min(n, i + step)) for i in range(0, n, step)]


def _terms(P, pos):
    dx = P[:, 0:1] - pos[None, :, 0]
    dy = P[:, 1:2] - pos[None, :, 1]
    return dx, dy, (dx * dx + dy * dy + P[:, 2:3] ** 2).sqrt()


def exact(case, seed):
    if case["kind"] not in ("eval", "train"):
        return None   # the result of a search depends on its decisions
    (B0, xyz, lam, up), = _inputs(case, seed)
    pos, b = _quadrature(case, B0)
    n, N = len(xyz), len(pos)
    if n * N > 7e9:
        return None
    P, lam, h = xyz.double(), lam.double(), case["h"]
    z = P[:, 2]
    B = torch.zeros(n, 3, dtype=torch.float64, device="cuda")
    G = torch.zeros(n, 3, 3, dtype=torch.float64, device="cuda")
    gB0 = torch.zeros(3, N, dtype=torch.float64, device="cuda")
    glam = torch.zeros_like(B)
    for k in _chunks(n, N):
        dx, dy, r = _terms(P[k], pos)
        zk = z[k, None]
        for p in range(3):
            l = lam[k, p, None]
            s, co = torch.sin(l * r), torch.cos(l * r)
            u = l * r * s + co
            phi = u / r ** 3
            B[k, p] = z[k] * (phi @ b[p])
            if case["grad"]:
                psi = (l * l * co - 3 * u / r ** 2) / r ** 3
                G[k, p, 0] = z[k] * ((psi * dx) @ b[p])
                G[k, p, 1] = z[k] * ((psi * dy) @ b[p])
                G[k, p, 2] = phi @ b[p] + z[k] ** 2 * (psi @ b[p])
            if case["kind"] == "train":
                g = up[k, p, None].double()
                gB0[p] += ((g * zk) * phi).sum(0) * (h * h / (2 * math.pi))
                glam[k, p] = up[k, p].double() * z[k] * lam[k, p] * ((co / r) @ b[p])
        if case["quad"] < 0:   # z / (2 pi r^3) integrated over the pixels, for the low points
            low = zk <= 2 * h
            area = torch.zeros_like(r)
            for sx in (-0.5, 0.5):
                for sy in (-0.5, 0.5):
                    a, e = sx * h - dx, sy * h - dy
                    area += (4 * sx * sy) * torch.atan(a * e / (zk * (a * a + e * e + zk * zk).sqrt()))
            B[k] += (low * (area / (h * h) - zk / r ** 3)) @ b.T
    if case["kind"] == "train":
        return {"B": B, "gB0": gB0.T.reshape(B0.shape[1], B0.shape[2], 3), "glam": glam}
    if not case["grad"]:
        return {"B": B}
    J = torch.stack([G[:, 2, 1] - G[:, 1, 2], G[:, 0, 2] - G[:, 2, 0], G[:, 1, 0] - G[:, 0, 1]], 1)
    nB = B.norm(dim=1)
    f = torch.linalg.cross(J, B).norm(dim=1) / (J.norm(dim=1) * nB)
    g = (G[:, 0, 0] + G[:, 1, 1] + G[:, 2, 2]).abs() * (h / 6) / nB
    return {"B": B, "gradB": G, "f": f, "g": g, "phi": f + g}
