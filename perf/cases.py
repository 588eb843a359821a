"""Performance cases: what a user of the library has it do, through its public calls.

The kinds of work (key "what"):

  layer       one application of a layer operator (or of a fused single plus
              double layer) on a prepared point set: the matvec of a user's own
              Krylov loop, boundary data for a field evaluation
  transpose   one application of a transposed operator (adjoint solves)
  batch       one application over many surfaces and right-hand sides
  solve       a whole Dirichlet-Neumann solve
  gradient    a solve with its adjoint gradients in kappa, gamma and the points
  field       velocity off the surface from the boundary data of a solve
  quadrature  quadrature points of a star-shaped surface

Surfaces, spacings and parameters are those of the tests, the benchmark and
the batched recipe: spheres, ellipsoids and star surfaces at h = 1/6 .. 1/128,
delta = 3 h, mu = 1, kappa in 1 .. 1e-2.  Densities are smooth fields of the
coordinates (pressures, velocities and tractions of a solve), or white noise
("normal", the hardest Krylov vectors).
"""
import math

import numpy as np
import torch

import paper_2110_10749_gb300 as ssd
from paper_2110_10749_gb300 import workloads

PREC = {"fp64": ssd.FP64, "fp32c": ssd.FP32C}
TRANSPOSED = {"laplace_SL": ssd.OP_LAPLACE_SL, "laplace_DL": ssd.OP_LAPLACE_DL,
              "stokes_SL": ssd.OP_STOKES_SL, "stokes_DL": ssd.OP_STOKES_DL}
# nominal flops of a far pair (an FMA is two, a reciprocal square root one)
PAIR_FLOPS = {"laplace_SL": 11, "laplace_DL": 17, "stokes_SL": 26, "stokes_DL": 31, "stokes_SLDL": 51,
              "laplace_SLDL": 19}
MU = 1.3
ALPHA, BETA = 0.7, -1.1

_ctx = None


def context():
    """The program's one library context."""
    global _ctx
    if _ctx is None:
        _ctx = ssd.Context(0)
    return _ctx


# --------------------------------------------------------------------- the cases
def listed():
    sphere = {"a": 1.0, "b": 1.0, "c": 1.0}
    e75 = {"a": 1.0, "b": 0.7, "c": 0.5}
    return [
        # the smallest set in use (h = 1/8, 1062 points) in the default precision: latency
        {"name": "sdl_fp64_1k", "what": "layer", "op": "stokes_DL", "h_inv": 8.0, "prec": "fp64",
         "density": "smooth", **sphere},
        # Darcy matvec of the h = 1/32 sphere (17070 points) in the default precision, on noise
        {"name": "ldl_fp64_17k", "what": "layer", "op": "laplace_DL", "h_inv": 32.0, "prec": "fp64",
         "density": "normal", **sphere},
        # fused matvec of the implicit slip on the thin ellipsoid (1742 points)
        {"name": "ssldl_fp64_2k", "what": "layer", "op": "stokes_SLDL", "h_inv": 16.0, "prec": "fp64",
         "density": "smooth", "a": 1.0, "b": 0.6, "c": 0.4},
        # right-hand side of the Stokes step at h = 1/96 (78106 points), FP64: the residual of refined solves
        {"name": "ssl_fp64_78k", "what": "layer", "op": "stokes_SL", "h_inv": 96.0, "prec": "fp64",
         "density": "smooth", **e75},
        # Stokes matvec of the h = 1/32 sphere in the fast precision
        {"name": "sdl_fp32c_17k", "what": "layer", "op": "stokes_DL", "h_inv": 32.0, "prec": "fp32c",
         "density": "smooth", **sphere},
        # the benchmark's dominant operator (h = 1/128, 138830 points)
        {"name": "sdl_fp32c_139k", "what": "layer", "op": "stokes_DL", "h_inv": 128.0, "prec": "fp32c",
         "density": "smooth", **e75},
        # adjoint Stokes matvec at h = 1/16 (4302 points)
        {"name": "sdlt_fp64_4k", "what": "transpose", "op": "stokes_DL", "h_inv": 16.0, "prec": "fp64",
         "density": "smooth", **sphere},
        # matvec of the batched recipe: 6 surfaces, 4 far fields
        {"name": "batch_fp32c_6x4", "what": "batch", "op": "stokes_SLDL", "stars": 5, "ellipsoids": 1, "nrhs": 4,
         "h_lo": 16.0, "h_hi": 32.0, "prec": "fp32c"},
        # plain FP64 solve of the smallest set, lagged slip
        {"name": "solve_fp64_1k", "what": "solve", "h_inv": 8.0, "kappa": 1.0, "gamma": 1.0, "prec": "fp64",
         "refine": 0, "tol": 1e-10, "inner_tol": 1e-11, **sphere},
        # mixed-precision solve with FP64 residuals at h = 1/32 (17070 points)
        {"name": "solve_refined_17k", "what": "solve", "h_inv": 32.0, "kappa": 1.0, "gamma": 0.1, "prec": "fp32c",
         "refine": 4, "tol": 1e-10, "inner_tol": 1e-11, **sphere},
        # value and all gradients on a star surface (shape optimisation)
        {"name": "gradient_star_1k", "what": "gradient", "star": 2, "h_inv": 8.0, "kappa": 0.1, "gamma": 0.5,
         "tol": 1e-11},
        # velocity at field points in a shell around the h = 1/32 sphere
        {"name": "field_17k_20k", "what": "field", "h_inv": 32.0, "targets": 20001, **sphere},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _ellipsoid(rng):
    return {"a": 1.0, "b": round(rng.uniform(0.55, 1.0), 3), "c": round(rng.uniform(0.4, 1.0), 3)}


def _area(c):
    p = 1.6075
    ab, ac, bc = (c["a"] * c["b"]) ** p, (c["a"] * c["c"]) ** p, (c["b"] * c["c"]) ** p
    return 4.0 * math.pi * ((ab + ac + bc) / 3.0) ** (1.0 / p)


def _h_inv(c, n):
    """1/h that gives about n points (17070 on the unit sphere at h = 1/32)."""
    return round(32.0 * math.sqrt(n / 17070.0 * 4.0 * math.pi / _area(c)), 3)


def draw(rng):
    kind = rng.choice(["layer", "layer", "layer", "layer", "transpose", "batch", "solve", "gradient", "field",
                       "quadrature"])
    if kind in ("layer", "transpose"):
        prec = rng.choice(["fp64", "fp64", "fp32c"])
        top = 20000.0 if kind == "transpose" else (70000.0 if prec == "fp64" else 130000.0)
        c = _ellipsoid(rng)
        ops = sorted(TRANSPOSED if kind == "transpose" else PAIR_FLOPS)
        return {"what": kind, "op": rng.choice(ops), "h_inv": _h_inv(c, _log(rng, 600.0, top)), "prec": prec,
                "density": rng.choice(["smooth", "smooth", "normal"]), **c}
    if kind == "batch":
        lo = round(_log(rng, 8.0, 16.0), 3)
        return {"what": kind, "op": rng.choice(["laplace_DL", "stokes_DL", "stokes_SLDL"]),
                "stars": rng.randint(1, 4), "ellipsoids": rng.randint(0, 2), "nrhs": rng.randint(1, 4), "h_lo": lo,
                "h_hi": round(lo * rng.uniform(1.2, 2.0), 3), "prec": rng.choice(["fp64", "fp32c"])}
    if kind == "solve":
        c = _ellipsoid(rng)
        refined = rng.random() < 0.5
        return {"what": kind, "h_inv": _h_inv(c, _log(rng, 700.0, 9000.0 if refined else 2500.0)),
                "kappa": round(_log(rng, 0.1, 1.0), 4), "gamma": round(_log(rng, 0.1, 1.0), 4),
                "prec": "fp32c" if refined else "fp64", "refine": 4 if refined else 0, "tol": 1e-10,
                "inner_tol": 1e-11, **c}
    if kind == "gradient":
        return {"what": kind, "star": rng.randint(0, 15), "h_inv": round(rng.uniform(5.5, 7.5), 3),
                "kappa": round(_log(rng, 0.1, 1.0), 4), "gamma": round(_log(rng, 0.1, 1.0), 4), "tol": 1e-11}
    if kind == "field":
        c = _ellipsoid(rng)
        return {"what": kind, "h_inv": _h_inv(c, _log(rng, 700.0, 20000.0)), "targets": int(_log(rng, 50.0, 20000.0)),
                **c}
    return {"what": kind, "h_inv": round(_log(rng, 10.0, 48.0), 3)}


# -------------------------------------------------------------------- preparation
class _State:
    """What a program keeps: handles are given back when it is dropped."""

    def __del__(self):
        for name in ("points", "batch"):
            held = getattr(self, name, None)
            if held is not None:
                try:
                    held.release()
                except Exception:
                    pass


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _field_of(xyz, comps, seed):
    """Smooth random fields of the coordinates, [comps][n]."""
    rng = np.random.default_rng(seed)
    x, y, z = xyz
    out = []
    for _ in range(comps):
        k, c = rng.uniform(-2.0, 2.0, (3, 3)), rng.normal(size=8)
        phase = [k[i, 0] * x + k[i, 1] * y + k[i, 2] * z for i in range(3)]
        out.append(c[0] * torch.sin(phase[0]) + c[1] * torch.cos(phase[1]) + c[2] * torch.exp(0.5 * phase[2])
                   + c[3] * x + c[4] * y + c[5] * z + c[6] * x * y + c[7])
    return torch.stack(out).contiguous()


def _density(case, xyz, comps, seed):
    if case.get("density", "smooth") == "normal":
        return torch.randn((comps, xyz.shape[1]), dtype=torch.float64, device="cuda", generator=_generator(seed))
    return _field_of(xyz, comps, seed)


def _surface_points(case):
    abc = (case["a"], case["b"], case["c"])
    return ssd.quadrature_points(context(), ssd.ELLIPSOID, abc, 1.0 / case["h_inv"])


def _direction(seed):
    v = np.random.default_rng(seed).normal(size=3)
    return tuple(float(t) for t in v / np.linalg.norm(v))


def _prepared(q):
    return ssd.Points(q["xyz"], q["nrm"], q["w"]).prepare(context())


def _comps(op):
    return 1 if op.startswith("laplace") else 3


def prepare(case, seed):
    s = _State()
    s.case, what = case, case["what"]
    ctx = context()
    if what == "quadrature":
        s.h, s.clm = 1.0 / case["h_inv"], workloads.star_coefficients(1000 + seed)
        return s
    if what == "batch":
        rng = np.random.default_rng([case["stars"], case["ellipsoids"]])
        sets, s.delta = [], []
        for k in range(case["stars"] + case["ellipsoids"]):
            h = 1.0 / rng.uniform(case["h_lo"], case["h_hi"])
            if k < case["stars"]:
                sets.append(ssd.quadrature_points(ctx, ssd.STAR, h=h, clm=workloads.star_coefficients(k)))
            else:
                sets.append(ssd.quadrature_points(ctx, ssd.ELLIPSOID, (1.0, 0.8, 0.6), h))
            s.delta.append(3.0 * h)
        s.offsets = np.concatenate([[0], np.cumsum([int(q["w"].numel()) for q in sets])])
        cat = {k: torch.cat([q[k] for q in sets], dim=-1).contiguous() for k in ("xyz", "nrm", "w")}
        s.batch = ssd.Batch(cat["xyz"], cat["nrm"], cat["w"], s.offsets, s.delta).prepare(ctx)
        nc = _comps(case["op"])
        s.d0 = torch.stack([_field_of(cat["xyz"], nc, [seed, r, 0]) for r in range(case["nrhs"])])
        s.d1 = torch.stack([_field_of(cat["xyz"], nc, [seed, r, 1]) for r in range(case["nrhs"])])
        return s
    if what == "gradient":
        q = ssd.quadrature_points(ctx, ssd.STAR, h=1.0 / case["h_inv"], clm=workloads.star_coefficients(case["star"]))
    else:
        q = _surface_points(case)
    s.delta = 3.0 / case["h_inv"]
    s.points = _prepared(q)
    if what in ("layer", "transpose"):
        nc = _comps(case["op"])
        s.d0 = _density(case, q["xyz"], nc, seed)
        s.d1 = _density(case, q["xyz"], nc, seed + 100003)
        if nc == 1:
            s.d0, s.d1 = s.d0[0].contiguous(), s.d1[0].contiguous()
    elif what == "solve":
        inner = ssd.krylov(case["inner_tol"], 256, 256, False, PREC[case["prec"]], deflate=True)
        s.prm = ssd.ddm_params(mu=1.0, kappa=case["kappa"], gamma=case["gamma"], uinf=_direction(seed),
                               delta=s.delta, theta=0.5 * case["kappa"], tol_outer=case["tol"], maxit_outer=128,
                               outer_gmres=True, traction_mode=ssd.TRACTION_BJS, inner=inner,
                               refine=case["refine"])
    elif what == "gradient":
        inner = ssd.krylov(0.1 * case["tol"], 400, 100, False, ssd.FP64, True)
        s.prm = ssd.ddm_params(mu=1.0, kappa=case["kappa"], gamma=case["gamma"], uinf=_direction(seed),
                               delta=s.delta, theta=1.0, tol_outer=case["tol"], maxit_outer=80, outer_gmres=True,
                               traction_mode=ssd.TRACTION_BJS, inner=inner, bjs_implicit=True)
    elif what == "field":
        s.f, s.u = _field_of(q["xyz"], 3, seed), _field_of(q["xyz"], 3, seed + 100003)
        t = torch.rand((3, case["targets"]), dtype=torch.float64, device="cuda", generator=_generator(seed)) * 2 - 1
        # field points in the shell 1.3 <= |y| <= 3 around the body
        s.targets = (t / t.norm(dim=0) * (1.3 + 1.7 * t.abs().amax(dim=0))).contiguous()
        s.uinf = _direction(seed)
    return s


# ---------------------------------------------------------------------------- run
def run(s):
    case, ctx = s.case, context()
    what = case["what"]
    if what == "layer":
        op, prec, P = case["op"], PREC[case["prec"]], s.points
        if op in ("laplace_SL", "laplace_DL", "stokes_DL"):
            return getattr(ssd, op)(ctx, P, s.delta, s.d0, prec)
        if op == "stokes_SL":
            return ssd.stokes_SL(ctx, P, s.delta, MU, s.d0, prec)
        if op == "stokes_SLDL":
            return ssd.stokes_SLDL(ctx, P, s.delta, MU, s.d1, s.d0, ALPHA, BETA, prec)
        return ssd.laplace_SLDL(ctx, P, s.delta, s.d1, s.d0, ALPHA, BETA, prec)
    if what == "transpose":
        return ssd.apply_transpose(ctx, s.points, TRANSPOSED[case["op"]], s.delta, s.d0, mu=MU,
                                   prec=PREC[case["prec"]])
    if what == "batch":
        op = {"laplace_DL": ssd.OP_LAPLACE_DL, "stokes_DL": ssd.OP_STOKES_DL,
              "stokes_SLDL": ssd.OP_STOKES_SLDL}[case["op"]]
        return ssd.batch_apply(ctx, s.batch, op, s.d0, s.d1 if case["op"] == "stokes_SLDL" else None, MU, ALPHA, BETA,
                               PREC[case["prec"]])
    if what == "solve":
        r = ssd.ddm_solve(ctx, s.points, s.prm)
        return {k: r[k] for k in ("q", "p", "u", "f", "drag")}
    if what == "gradient":
        value, grad, (gx, gn, gw), _ = ssd.ddm_gradient_geometry(ctx, s.points, s.prm, ssd.FUNC_DRAG)
        return {"value": value, "grad": grad, "gx": gx, "gn": gn, "gw": gw}
    if what == "field":
        return ssd.stokes_velocity_field(ctx, s.points, 1.0, s.uinf, s.f, s.u, s.targets)
    return ssd.quadrature_points(ctx, ssd.STAR, h=s.h, clm=s.clm)


# --------------------------------------------------------------------------- work
def _points_of(case):
    if case["what"] in ("gradient", "quadrature"):
        return 17070.0 * (case["h_inv"] / 32.0) ** 2
    return 17070.0 * (case["h_inv"] / 32.0) ** 2 * _area(case) / (4.0 * math.pi)


def work(case):
    """Each input read once and each output written once; nominal pair flops.
    A solve counts the applications that its equations cannot do without: two
    right-hand sides and, for each of three sweeps, five steps of both local
    solves; a gradient three such solves."""
    what = case["what"]
    if what == "batch":
        k, nc = case["stars"] + case["ellipsoids"], _comps(case["op"])
        n = 17070.0 * (0.5 * (case["h_lo"] + case["h_hi"]) / 32.0) ** 2
        dens = 3 if case["op"] == "stokes_SLDL" else 2
        return {"bytes": 8.0 * k * n * (7 + case["nrhs"] * nc * dens),
                "flops": k * case["nrhs"] * n * n * PAIR_FLOPS[case["op"]]}
    n = _points_of(case)
    if what in ("layer", "transpose"):
        nc = _comps(case["op"])
        dens = 3 if case["op"].endswith("SLDL") else 2
        return {"bytes": 8.0 * n * (7 + nc * dens), "flops": n * n * PAIR_FLOPS[case["op"]]}
    if what == "solve":
        return {"bytes": 8.0 * n * 15, "flops": 3.0 * n * n * (11 + 26 + 5 * (17 + 31))}
    if what == "gradient":
        return {"bytes": 8.0 * n * 14, "flops": 9.0 * n * n * (11 + 26 + 5 * (17 + 51))}
    if what == "field":
        m = float(case["targets"])
        return {"bytes": 8.0 * (13 * n + 6 * m), "flops": n * m * 51}
    # one sign test of the level set per grid step and line, three axes
    lines = 3.0 * (2.4 * case["h_inv"]) ** 2
    return {"bytes": 8.0 * n * 9, "flops": lines * 160.0 * 100.0}


# -------------------------------------------------------- the same in plain torch
_NSER = 40


def _series(i):
    """Taylor coefficients of s_i(rho) / rho^p in t = rho^2 (p = 1, 3, 3, 5)."""
    q = {1: (5 / 3, -2 / 3, 0.0, 0.0), 2: (-1.0, 2 / 3, 0.0, 0.0), 3: (-1.0, 14 / 3, -4 / 3, 0.0),
         4: (-1.0, -6 / 9, 4.0, -8 / 9)}[i]
    skip = {1: 0, 2: 1, 3: 1, 4: 2}[i]
    c = []
    for k in range(skip, skip + _NSER):
        v = (-1.0) ** k / (math.factorial(k) * (2 * k + 1))
        v += sum(q[m] * (-1.0) ** (k - m) / math.factorial(k - m) for m in range(4) if m <= k)
        c.append(2.0 / math.sqrt(math.pi) * v)
    return c


def _sigma(i, t):
    """s_i / rho^p: the series below rho = 1, the closed form of the paper above."""
    p = {1: 1, 2: 3, 3: 3, 4: 5}[i]
    ts = torch.clamp(t, max=1.0)
    ser = torch.zeros_like(t)
    for c in reversed(_series(i)):
        ser = ser * ts + c
    tc = torch.clamp(t, min=1.0)
    rho = torch.sqrt(tc)
    te = torch.clamp(tc, max=100.0)
    poly = {1: lambda: -(2 * te - 5) / 3, 2: lambda: (2 * te - 3) / 3, 3: lambda: -(4 * te * te - 14 * te + 3) / 3,
            4: lambda: -(8 * te ** 3 - 36 * te * te + 6 * te + 9) / 9}[i]()
    s = torch.erf(rho) + 2.0 / math.sqrt(math.pi) * torch.sqrt(te) * poly * torch.exp(-te)
    return torch.where(t < 1.0, ser, s / rho ** p)


def _rows(kind, xyz, nrm, w, delta, mu, rows, dens):
    """Rows of an operator applied to dens [c][n]: [c][len(rows)]."""
    d = xyz[:, rows, None] - xyz[:, None, :]
    t = (d * d).sum(0) / (delta * delta)
    if kind == "laplace_SL":
        return -(_sigma(1, t) / (4 * math.pi * delta)) @ (w * dens[0])[:, None]
    if kind == "laplace_DL":
        k = torch.einsum("aij,aj->ij", d, nrm * w) * _sigma(2, t) / (-4 * math.pi * delta ** 3)
        return (k * (dens[0][None, :] - dens[0][rows, None])).sum(1)[:, None]
    if kind == "stokes_SL":
        f = w * dens
        b = torch.einsum("aij,aj->ij", d, f) * _sigma(3, t) / delta ** 3
        s1 = _sigma(1, t) / delta
        return ((s1 @ f.T).T + torch.einsum("aij,ij->ai", d, b)).T / (8 * math.pi * mu)
    du = (torch.einsum("aij,aj->ij", d, dens) - torch.einsum("aij,ai->ij", d, dens[:, rows]))
    b = du * torch.einsum("aij,aj->ij", d, nrm * w) * _sigma(4, t) * (6 / (8 * math.pi) / delta ** 5)
    return torch.einsum("aij,ij->ai", d, b).T


def _transposed_rows(kind, xyz, nrm, w, delta, mu, rows, v):
    d = xyz[:, rows, None] - xyz[:, None, :]
    t = (d * d).sum(0) / (delta * delta)
    if kind == "laplace_SL":
        return -w[rows, None] * ((_sigma(1, t) / (4 * math.pi * delta)) @ v[0][:, None])
    if kind == "stokes_SL":
        b = torch.einsum("aij,aj->ij", d, v) * _sigma(3, t) / delta ** 3
        out = ((_sigma(1, t) / delta) @ v.T).T + torch.einsum("aij,ij->ai", d, b)
        return (w[rows] * out).T / (8 * math.pi * mu)
    m = nrm * w
    at, aj = torch.einsum("aij,ai->ij", d, m[:, rows]), torch.einsum("aij,aj->ij", d, m)
    if kind == "laplace_DL":
        k = _sigma(2, t) / (4 * math.pi * delta ** 3)
        return (k * (at * v[0][None, :] + aj * v[0][rows, None])).sum(1)[:, None]
    vj, vt = torch.einsum("aij,aj->ij", d, v), torch.einsum("aij,ai->ij", d, v[:, rows])
    b = (at * vj + aj * vt) * _sigma(4, t) * (-6 / (8 * math.pi) / delta ** 5)
    return torch.einsum("aij,ij->ai", d, b).T


def _all_rows(fn, n, comps):
    """fn over blocks of rows whose temporaries stay around a gigabyte."""
    step = max(1, min(n, int(8e6 / n)))
    out = torch.empty((comps, n), dtype=torch.float64, device="cuda")
    for k in range(0, n, step):
        rows = torch.arange(k, min(k + step, n), device="cuda")
        out[:, rows] = fn(rows).T
    return out


def _apply_plain(op, xyz, nrm, w, delta, d0, d1):
    nc = _comps(op)
    base = "laplace" if nc == 1 else "stokes"
    n = w.numel()
    if op.endswith("SLDL"):
        sl = _all_rows(lambda r: _rows(base + "_SL", xyz, nrm, w, delta, MU, r, d1), n, nc)
        dl = _all_rows(lambda r: _rows(base + "_DL", xyz, nrm, w, delta, MU, r, d0), n, nc)
        return ALPHA * sl + BETA * dl
    return _all_rows(lambda r: _rows(op, xyz, nrm, w, delta, MU, r, d0), n, nc)


def _dense(xyz, nrm, w, delta):
    """Dense L, D^L, M (mu = 1) and D^S on component-major vectors."""
    n = w.numel()
    d = xyz[:, :, None] - xyz[:, None, :]
    t = (d * d).sum(0) / (delta * delta)
    m = nrm * w
    dn = torch.einsum("aij,aj->ij", d, m)
    L = -_sigma(1, t) * w / (4 * math.pi * delta)
    DL = dn * _sigma(2, t) / (-4 * math.pi * delta ** 3)
    DL = DL - torch.diag(DL.sum(1))
    s1, s3 = _sigma(1, t) / delta, _sigma(3, t) / delta ** 3
    k = dn * _sigma(4, t) * (6 / (8 * math.pi) / delta ** 5)
    eye = torch.eye(3, dtype=torch.float64, device=w.device)
    M = (eye[:, None, :, None] * s1[None, :, None, :] + torch.einsum("aij,bij,ij->aibj", d, d, s3)) * w / (8 * math.pi)
    K = torch.einsum("aij,bij,ij->aibj", d, d, k)
    own = K.sum(3)                                  # [a][i][b]
    K = K - torch.einsum("aib,ij->aibj", own, torch.eye(n, dtype=torch.float64, device=w.device))
    return L, DL, M.reshape(3 * n, 3 * n), K.reshape(3 * n, 3 * n)


def _dense_solve(xyz, nrm, w, delta, kappa, gamma, uinf):
    """The fixed point of the Dirichlet-Neumann sweeps by one dense solve."""
    n = w.numel()
    L, DL, M, DS = _dense(xyz, nrm, w, delta)
    one = torch.ones(n, dtype=torch.float64, device=w.device)
    W = w.sum()
    mean = torch.outer(one, w) / W
    G = torch.linalg.solve(mean - DL, L / kappa)
    G = G - mean @ G                                # q -> p, zero weighted mean
    N = torch.cat([torch.diag(nrm[a]) for a in range(3)])             # p -> p n
    T = torch.eye(3 * n, dtype=torch.float64, device=w.device) - N @ N.T
    nv = nrm.reshape(-1)
    A = torch.eye(3 * n, dtype=torch.float64, device=w.device) - DS + torch.outer(nv, (nrm * w).reshape(-1)) / W
    c = gamma / math.sqrt(kappa) if not torch.is_tensor(kappa) else gamma / torch.sqrt(kappa)
    rhs = torch.repeat_interleave(torch.tensor(uinf, dtype=torch.float64, device=w.device), n)
    u = torch.linalg.solve(A + M @ (c * T - N @ (G @ N.T)), rhs)
    q = N.T @ u
    p = G @ q
    f = -(N @ p) + c * (T @ u)
    return q, p, u.reshape(3, n), f.reshape(3, n)


def exact(case, seed):
    what = case["what"]
    if what == "quadrature" or (what == "solve" and _points_of(case) > 4000):
        return None
    s = prepare(case, seed)
    if what == "batch":
        B, out = s.batch, []
        for r in range(case["nrhs"]):
            parts = []
            for k, delta in enumerate(s.delta):
                a, b = int(s.offsets[k]), int(s.offsets[k + 1])
                parts.append(_apply_plain(case["op"], B.xyz[:, a:b], B.nrm[:, a:b], B.w[a:b], delta,
                                          s.d0[r][:, a:b], s.d1[r][:, a:b]))
            out.append(torch.cat(parts, dim=1))
        return torch.stack(out)
    P = s.points
    xyz, nrm, w = P.xyz, P.nrm, P.w
    if what in ("layer", "transpose"):
        nc = _comps(case["op"])
        d0, d1 = s.d0.reshape(nc, -1), s.d1.reshape(nc, -1)
        if what == "layer":
            out = _apply_plain(case["op"], xyz, nrm, w, s.delta, d0, d1)
        else:
            out = _all_rows(lambda r: _transposed_rows(case["op"], xyz, nrm, w, s.delta, MU, r, d0), P.n, nc)
        return out if nc == 3 else out[0]
    if what == "solve":
        q, p, u, f = _dense_solve(xyz, nrm, w, s.delta, case["kappa"], case["gamma"], list(s.prm.uinf))
        return {"q": q, "p": p, "u": u, "f": f, "drag": (f @ w).cpu().numpy()}
    if what == "gradient":
        x, m, v = (t.clone().requires_grad_() for t in (xyz, nrm, w))
        lk = torch.tensor(math.log(case["kappa"]), dtype=torch.float64, device="cuda", requires_grad=True)
        gm = torch.tensor(case["gamma"], dtype=torch.float64, device="cuda", requires_grad=True)
        e = torch.tensor(list(s.prm.uinf), dtype=torch.float64, device="cuda")
        J = e @ (_dense_solve(x, m, v, s.delta, torch.exp(lk), gm, list(s.prm.uinf))[3] @ v)
        J.backward()
        return {"value": float(J), "grad": np.array([float(lk.grad), float(gm.grad)]), "gx": x.grad, "gn": m.grad,
                "gw": v.grad}
    # field: bare kernels at points off the surface
    out = torch.empty_like(s.targets)
    step = max(1, int(8e6 / P.n))
    for k in range(0, s.targets.shape[1], step):
        d = s.targets[:, k:k + step, None] - xyz[:, None, :]
        r = torch.sqrt((d * d).sum(0))
        f = w * s.f
        sl = ((1 / r) @ f.T).T + torch.einsum("aij,ij->ai", d, torch.einsum("aij,aj->ij", d, f) / r ** 3)
        b = torch.einsum("aij,aj->ij", d, s.u) * torch.einsum("aij,aj->ij", d, nrm * w) / r ** 5
        dl = torch.einsum("aij,ij->ai", d, b)
        out[:, k:k + step] = sl / (-8 * math.pi) + dl * (6 / (8 * math.pi))
    return out + torch.tensor(s.uinf, dtype=torch.float64, device="cuda")[:, None]
