"""The FP64 paths beside the fixed-point kernel's main one.  Point sets over 256
delta across run in double precision: the direct kernel with and without its launch
order, the plan with far block pairs, a batch with one such surface.  Densities
without a common scale run in double inside the fixed-point kernel: on a plan (its two
launches), on sets of 6000 points and more, on one surface of a batch.  Tolerance
1e-12 relative, as for every FP64 operator; the adjoint identity to 1e-12 of the
product of the norms."""
import numpy as np
import pytest

import oracle
from oracle import quadrature as Q

pytestmark = pytest.mark.gpu

MU, ALPHA, BETA, DELTA = 1.3, 0.7, -1.1, 0.5
TOL = 1e-12


def spheres(k, spacing, m=512):
    """k unit spheres of m points on the corners of a cube (one of 100 points less): in the
    spatial order m / 512 blocks each, far apart."""
    q = Q.sphere_points(1.0, 1 / 6 if m <= 512 else 1 / 8)
    pick = np.linspace(0, q["w"].size - 1, m).astype(int)
    p = {a: q[a][..., pick] for a in q if a in ("xyz", "nrm", "w")}
    x = [p["xyz"] + spacing * np.array([[i >> 2 & 1], [i >> 1 & 1], [i & 1]]) for i in range(k)]
    n = k * m - 100
    return {"xyz": np.ascontiguousarray(np.concatenate(x, axis=1)[:, :n]),
            "nrm": np.ascontiguousarray(np.tile(p["nrm"], (1, k))[:, :n]), "w": np.tile(p["w"], k)[:n]}


def densities(n, seed):
    rng = np.random.default_rng(seed)
    return rng.normal(size=n), rng.normal(size=(3, n)), rng.normal(size=n), rng.normal(size=(3, n))


def reference(p, g, v, g2, v2):
    r = {"LSL": oracle.laplace_sl(p, DELTA, g), "LDL": oracle.laplace_dl(p, DELTA, g),
         "SSL": oracle.stokes_sl(p, DELTA, MU, v), "SDL": oracle.stokes_dl(p, DELTA, v)}
    r["LSLDL"] = ALPHA * oracle.laplace_sl(p, DELTA, g2) + BETA * r["LDL"]
    r["SSLDL"] = ALPHA * oracle.stokes_sl(p, DELTA, MU, v2) + BETA * r["SDL"]
    return r


def device(ssd, ctx, P, g, v, g2, v2):
    import torch
    g, v, g2, v2 = (torch.as_tensor(a, device="cuda") for a in (g, v, g2, v2))
    o = {"LSL": ssd.laplace_SL(ctx, P, DELTA, g), "LDL": ssd.laplace_DL(ctx, P, DELTA, g),
         "SSL": ssd.stokes_SL(ctx, P, DELTA, MU, v), "SDL": ssd.stokes_DL(ctx, P, DELTA, v),
         "SSLDL": ssd.stokes_SLDL(ctx, P, DELTA, MU, v2, v, ALPHA, BETA),
         "LSLDL": ssd.laplace_SLDL(ctx, P, DELTA, g2, g, ALPHA, BETA)}
    return {k: t.cpu().numpy() for k, t in o.items()}


def transposes(ssd, ctx, P, g, v):
    import torch
    return {k: ssd.apply_transpose(ctx, P, op, DELTA, torch.as_tensor(x, device="cuda"), mu=MU).cpu().numpy()
            for k, op, x in (("LDL", ssd.OP_LAPLACE_DL, g), ("SDL", ssd.OP_STOKES_DL, v))}


def close(out, ref):
    for k, b in ref.items():
        assert np.linalg.norm(out[k] - b) <= TOL * np.linalg.norm(b), k


def planned(ctx, call):
    """Packing, near items, far items and epilogue are four launches, a direct application three."""
    call()
    before = ctx.launch_count()
    call()
    return ctx.launch_count() - before == 4


def context(ssd, monkeypatch, **env):
    for k, x in env.items():
        monkeypatch.setenv(k, x)
    ctx = ssd.Context(0)
    for k in env:
        monkeypatch.delenv(k)
    return ctx


def test_points_over_256_delta_across(gpu_ctx, monkeypatch):
    import torch

    import paper_2110_10749_gb300 as ssd
    p = spheres(8, 130.0)                     # extent 132, 264 delta
    n = p["w"].size
    dens = densities(n, 1)
    ref = reference(p, *dens)
    P = ssd.Points.from_numpy(p).prepare(gpu_ctx)
    close(device(ssd, gpu_ctx, P, *dens), ref)
    tv = torch.as_tensor(dens[1], device="cuda")
    assert planned(gpu_ctx, lambda: ssd.stokes_DL(gpu_ctx, P, DELTA, tv))
    # transposes (direct) by the adjoint identity
    t = transposes(ssd, gpu_ctx, P, dens[2], dens[3])
    for k, x, y in (("LDL", dens[0], dens[2]), ("SDL", dens[1], dens[3])):
        assert abs((ref[k] * y).sum() - (t[k] * x).sum()) <= TOL * np.linalg.norm(ref[k]) * np.linalg.norm(y), k
    P.release()
    # the direct kernels, in near-first order and in plain order: the same sums, bit for bit
    out = []
    for lpt in ("1", "0"):
        ctx = context(ssd, monkeypatch, SSD_PAIR_SYM="0", SSD_PAIR_LPT=lpt)
        P = ssd.Points.from_numpy(p).prepare(ctx)
        out.append(device(ssd, ctx, P, *dens))
        assert not planned(ctx, lambda: ssd.stokes_DL(ctx, P, DELTA, tv))
        P.release()
        ctx.close()
    close(out[0], ref)
    for k in ref:
        assert np.array_equal(out[0][k], out[1][k]), k


def test_batch_with_a_surface_over_256_delta_across(gpu_ctx):
    import torch

    import paper_2110_10749_gb300 as ssd
    pts = [spheres(1, 0.0), spheres(2, 140.0), spheres(1, 0.0)]
    offs = np.concatenate([[0], np.cumsum([p["w"].size for p in pts])])
    B = ssd.Batch.from_numpy(pts, [DELTA] * 3).prepare(gpu_ctx)
    g, v, g2, v2 = (a[None] for a in densities(offs[-1], 2))
    T = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    kw = dict(mu=MU, alpha=ALPHA, beta=BETA)
    out = {"LSL": ssd.batch_apply(gpu_ctx, B, ssd.OP_LAPLACE_SL, T(g), **dict(kw, alpha=1.0, beta=1.0)),
           "LDL": ssd.batch_apply(gpu_ctx, B, ssd.OP_LAPLACE_DL, T(g), **dict(kw, alpha=1.0, beta=1.0)),
           "SSL": ssd.batch_apply(gpu_ctx, B, ssd.OP_STOKES_SL, T(v), **dict(kw, alpha=1.0, beta=1.0)),
           "SDL": ssd.batch_apply(gpu_ctx, B, ssd.OP_STOKES_DL, T(v), **dict(kw, alpha=1.0, beta=1.0)),
           "SSLDL": ssd.batch_apply(gpu_ctx, B, ssd.OP_STOKES_SLDL, T(v), T(v2), **kw),
           "LSLDL": ssd.batch_apply(gpu_ctx, B, ssd.OP_LAPLACE_SLDL, T(g), T(g2), **kw)}
    for s, p in enumerate(pts):
        sl = slice(offs[s], offs[s + 1])
        ref = reference(p, *(np.ascontiguousarray(a[0][..., sl]) for a in (g, v, g2, v2)))
        close({k: t.cpu().numpy()[0][..., sl] for k, t in out.items()}, ref)
    B.release()


@pytest.mark.parametrize("m", [512, 1024])    # 3996 points; 8092, over 6000
def test_densities_without_a_common_scale_on_large_sets(gpu_ctx, monkeypatch, m):
    import torch

    import paper_2110_10749_gb300 as ssd
    p = spheres(8, 20.0, m)
    n = p["w"].size
    dens = densities(n, 3)
    ref = reference(p, *dens)
    direct = context(ssd, monkeypatch, SSD_PAIR_SYM="0")
    for ctx, plan in ((gpu_ctx, True), (direct, False)):
        P = ssd.Points.from_numpy(p).prepare(ctx)
        tv = torch.as_tensor(dens[1], device="cuda")
        assert planned(ctx, lambda: ssd.stokes_DL(ctx, P, DELTA, tv)) == plan
        big = device(ssd, ctx, P, *(1e200 * a for a in dens))
        # norms in units of 1e200, where they do not overflow
        close({q: a / 1e200 for q, a in big.items()}, ref)
        t = transposes(ssd, ctx, P, 1e200 * dens[2], 1e200 * dens[3])
        for q, x, y in (("LDL", dens[0], dens[2]), ("SDL", dens[1], dens[3])):
            assert abs((ref[q] * y).sum() - (t[q] / 1e200 * x).sum()) <= \
                TOL * np.linalg.norm(ref[q]) * np.linalg.norm(y), q
        bad = [a.copy() for a in dens]
        for a in bad:
            a[..., n // 2] = np.nan
        for q, a in device(ssd, ctx, P, *bad).items():
            assert np.isnan(a).all(), q
        P.release()
    direct.close()


@pytest.mark.parametrize("value", [1e200, float("nan")])
def test_one_surface_of_a_batch_without_a_common_scale(gpu_ctx, value):
    import torch

    import paper_2110_10749_gb300 as ssd
    pts = [spheres(1, 0.0), spheres(2, 4.0), spheres(1, 0.0)]
    offs = np.concatenate([[0], np.cumsum([p["w"].size for p in pts])])
    B = ssd.Batch.from_numpy(pts, [DELTA] * 3).prepare(gpu_ctx)
    _, v, _, f = densities(offs[-1], 4)
    sv, sf = v.copy(), f.copy()
    for a in (sv, sf):
        a[:, offs[1]:offs[2]] *= value
    T = lambda a: torch.as_tensor(a[None], device="cuda")
    out = ssd.batch_apply(gpu_ctx, B, ssd.OP_STOKES_SLDL, T(sv), T(sf), mu=MU, alpha=ALPHA,
                          beta=BETA).cpu().numpy()[0]
    for s, p in enumerate(pts):
        sl = slice(offs[s], offs[s + 1])
        x, y = np.ascontiguousarray(v[:, sl]), np.ascontiguousarray(f[:, sl])
        ref = ALPHA * oracle.stokes_sl(p, DELTA, MU, y) + BETA * oracle.stokes_dl(p, DELTA, x)
        if s == 1 and value != value:
            assert np.isnan(out[:, sl]).all()
        else:
            close({"SSLDL": out[:, sl] / (value if s == 1 else 1.0)}, {"SSLDL": ref})
    B.release()
