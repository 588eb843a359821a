"""The FP64 operators on the fixed-point kernel: sizes around its tiles (chunks
of 32 sources, staged tiles of 128, CTAs of 256 targets), density scales, the
edge of its range (extent 256 delta; beyond it the generic kernel runs) and
densities it hands to double precision (not finite, or without a common
scale).  Tolerance 1e-12 relative, as for every FP64 operator."""
import numpy as np
import pytest

import oracle
from oracle import quadrature as Q

pytestmark = pytest.mark.gpu

MU, ALPHA, BETA = 1.3, 0.7, -1.1
TOL = 1e-12


def subset(full, n):
    k = np.linspace(0, full["w"].size - 1, n).astype(int)
    return {q: np.ascontiguousarray(full[q][..., k]) for q in ("xyz", "nrm", "w")}


def dense(p, d, g, v, g2, v2):
    """Every operator from the oracle's dense matrices."""
    A = {k: oracle.operator_matrix(p, d, k, mu=MU) for k in ("L", "DL", "M", "DS")}
    n = p["w"].size
    S = lambda M, x: (M @ x.reshape(-1)).reshape(3, n)
    return {"LSL": A["L"] @ g, "LDL": A["DL"] @ g, "SSL": S(A["M"], v), "SDL": S(A["DS"], v),
            "SSLDL": ALPHA * S(A["M"], v2) + BETA * S(A["DS"], v), "LSLDL": ALPHA * A["L"] @ g2 + BETA * A["DL"] @ g,
            "LSLT": A["L"].T @ g, "LDLT": A["DL"].T @ g, "SSLT": S(A["M"].T, v), "SDLT": S(A["DS"].T, v)}


def device(ssd, ctx, P, d, g, v, g2, v2):
    import torch
    g, v, g2, v2 = (torch.as_tensor(a, device="cuda") for a in (g, v, g2, v2))
    o = {"LSL": ssd.laplace_SL(ctx, P, d, g), "LDL": ssd.laplace_DL(ctx, P, d, g), "SSL": ssd.stokes_SL(ctx, P, d, MU, v),
         "SDL": ssd.stokes_DL(ctx, P, d, v), "SSLDL": ssd.stokes_SLDL(ctx, P, d, MU, v2, v, ALPHA, BETA),
         "LSLDL": ssd.laplace_SLDL(ctx, P, d, g2, g, ALPHA, BETA)}
    for k, op, x in (("LSLT", ssd.OP_LAPLACE_SL, g), ("LDLT", ssd.OP_LAPLACE_DL, g), ("SSLT", ssd.OP_STOKES_SL, v),
                     ("SDLT", ssd.OP_STOKES_DL, v)):
        o[k] = ssd.apply_transpose(ctx, P, op, d, x, mu=MU)
    return {k: t.cpu().numpy() for k, t in o.items()}


def close(out, ref, tol=TOL):
    for k, b in ref.items():
        scale = np.linalg.norm(b)
        assert np.linalg.norm(out[k] - b) <= tol * scale, (k, np.linalg.norm(out[k] - b), scale)


@pytest.fixture(scope="module")
def cloud():
    return Q.ellipsoid_points((1.0, 0.7, 0.5), 1 / 14, center=(0.1, -0.2, 3.0))


@pytest.mark.parametrize("n", [1, 2, 31, 33, 129, 256, 257, 513])
def test_sizes_around_the_tiles(gpu_ctx, cloud, n):
    import paper_2110_10749_gb300 as ssd
    p = subset(cloud, n)
    rng = np.random.default_rng(n)
    dens = rng.normal(size=n), rng.normal(size=(3, n)), rng.normal(size=n), rng.normal(size=(3, n))
    for d in (0.4, 0.05):
        ref = dense(p, d, *dens)
        P = ssd.Points.from_numpy(p)
        for prepared in (False, True):
            if prepared:
                P.prepare(gpu_ctx)
            close(device(ssd, gpu_ctx, P, d, *dens), ref)
        P.release()


@pytest.mark.parametrize("ratio", [255.0, 257.0])
def test_edge_of_the_range(gpu_ctx, cloud, ratio):
    # extent 2 (the long axis): the fixed-point kernel up to 256 delta, the generic one beyond
    import paper_2110_10749_gb300 as ssd
    p = subset(cloud, 300)
    ext = max(p["xyz"].max(axis=1) - p["xyz"].min(axis=1))
    d = ext / ratio
    rng = np.random.default_rng(2)
    dens = rng.normal(size=300), rng.normal(size=(3, 300)), rng.normal(size=300), rng.normal(size=(3, 300))
    P = ssd.Points.from_numpy(p).prepare(gpu_ctx)
    close(device(ssd, gpu_ctx, P, d, *dens), dense(p, d, *dens))
    P.release()


@pytest.mark.parametrize("scale,scale2", [(1e-100, 1e-100), (1e100, 1e90), (1.0, 0.0), (0.0, 1.0), (1e-20, 1e20),
                                          (1e200, 1e200)])
def test_density_scales(gpu_ctx, cloud, scale, scale2):
    # 1e200 has no common scale in the kernel's range: double precision inside the same launch
    import paper_2110_10749_gb300 as ssd
    n, d = 300, 0.3
    p = subset(cloud, n)
    rng = np.random.default_rng(4)
    dens = (scale * rng.normal(size=n), scale * rng.normal(size=(3, n)), scale2 * rng.normal(size=n),
            scale2 * rng.normal(size=(3, n)))
    P = ssd.Points.from_numpy(p).prepare(gpu_ctx)
    top = max(scale, scale2)
    # in units of 1e100 where the norm would overflow
    unit = 1e100 if top > 1e150 else 1.0
    out = device(ssd, gpu_ctx, P, d, *dens)
    ref = dense(p, d, *(a / unit for a in dens))
    close({k: a / unit for k, a in out.items()}, ref)
    P.release()


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_non_finite_densities_reach_every_target(gpu_ctx, cloud, value):
    import paper_2110_10749_gb300 as ssd
    n, d = 300, 0.3
    p = subset(cloud, n)
    rng = np.random.default_rng(6)
    g, v = rng.normal(size=n), rng.normal(size=(3, n))
    g[17] = value
    v[1, 17] = value
    P = ssd.Points.from_numpy(p).prepare(gpu_ctx)
    out = device(ssd, gpu_ctx, P, d, g, v, g, v)
    for k, a in out.items():
        assert not np.isfinite(a).any(), k
    P.release()


def test_batch_mixes_sizes_and_scales(gpu_ctx, cloud):
    import torch
    import paper_2110_10749_gb300 as ssd
    pts = [subset(cloud, n) for n in (5, 300, 513)]
    deltas = [0.5, 0.3, 0.2]
    B = ssd.Batch.from_numpy(pts, deltas).prepare(gpu_ctx)
    offs = np.concatenate([[0], np.cumsum([p["w"].size for p in pts])])
    rng = np.random.default_rng(8)
    nrhs = 2
    v, f = (rng.normal(size=(nrhs, 3, offs[-1])) for _ in range(2))
    for r, s in ((0, 1e-30), (1, 1e30)):    # every system has a scale of its own
        v[r] *= s
        f[r] *= s
        v[r][:, offs[1]:offs[2]] *= 1e-40
        f[r][:, offs[1]:offs[2]] *= 1e-40
    out = ssd.batch_apply(gpu_ctx, B, ssd.OP_STOKES_SLDL, torch.as_tensor(v, device="cuda"),
                          torch.as_tensor(f, device="cuda"), mu=MU, alpha=ALPHA, beta=BETA).cpu().numpy()
    for r in range(nrhs):
        for k, p in enumerate(pts):
            sl = slice(offs[k], offs[k + 1])
            x, y = np.ascontiguousarray(v[r][:, sl]), np.ascontiguousarray(f[r][:, sl])
            ref = ALPHA * oracle.stokes_sl(p, deltas[k], MU, y) + BETA * oracle.stokes_dl(p, deltas[k], x)
            assert np.linalg.norm(out[r][:, sl] - ref) <= TOL * np.linalg.norm(ref), (r, k)
    B.release()


def test_one_layout_serves_several_radii(gpu_ctx, cloud):
    # grid positions are kept per layout and radius
    import paper_2110_10749_gb300 as ssd
    n = 300
    p = subset(cloud, n)
    rng = np.random.default_rng(12)
    dens = rng.normal(size=n), rng.normal(size=(3, n)), rng.normal(size=n), rng.normal(size=(3, n))
    P = ssd.Points.from_numpy(p).prepare(gpu_ctx)
    for d in (0.4, 0.1, 0.1, 0.4):
        close(device(ssd, gpu_ctx, P, d, *dens), dense(p, d, *dens))
    P.release()
