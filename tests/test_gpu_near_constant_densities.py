"""FP64 double layers of densities that are nearly constant: the layers see differences
only, so the result belongs to the variation, whatever the constant, and a constant in
a fused layer leaves the single layer its digits.  Each is compared with the operator
on the variation alone, tolerance 1e-12 as for every FP64 operator.  The constants and
variations are such that their sums are exact (multiples of 2^-40 for components that
have both), and so are the records of these operators, which scale densities by 1; the
fused Stokes layers, whose records carry a constant of the kernel, take constants
only.  Small sets, grouped and not, a plan, plain points, a batch."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _round(v):
    import torch
    return torch.round(v * 2.0 ** 40) * 2.0 ** -40


def _data(ctx, h, scale):
    """Points, constant and varying densities, a single-layer density of that scale."""
    import torch

    import paper_2110_10749_gb300 as ssd
    q = ssd.quadrature_points(ctx, ssd.ELLIPSOID, (1.0, 0.8, 0.6), h)
    x = q["xyz"]
    var = scale * torch.sin(3.0 * x)
    var[0] = _round(var[0])                        # beside the constant 1
    var[1] = 0.0
    const = torch.zeros_like(x)
    const[0], const[1] = 1.0, -0.7
    f = (scale * torch.cos(2.0 * x)).contiguous()
    return q, const, var, f


def _close(a, b):
    assert float((a - b).norm()) <= 1e-12 * float(b.norm())


@pytest.mark.parametrize("h", [1 / 6, 1 / 12, 1 / 20, 1 / 40])
@pytest.mark.parametrize("scale", [1e-2, 1e-6])
@pytest.mark.parametrize("prepared", [False, True])
def test_layers_of_a_constant_and_a_variation(gpu_ctx, h, scale, prepared):
    import paper_2110_10749_gb300 as ssd
    q, const, var, f = _data(gpu_ctx, h, scale)
    d = 3 * h
    P = ssd.Points(q["xyz"], q["nrm"], q["w"])
    if prepared:
        P.prepare(gpu_ctx)
    u = (const + var).contiguous()
    p, vp, g = u[0].contiguous(), var[0].contiguous(), f[0].contiguous()
    _close(ssd.stokes_DL(gpu_ctx, P, d, u), ssd.stokes_DL(gpu_ctx, P, d, var))
    _close(ssd.laplace_DL(gpu_ctx, P, d, p), ssd.laplace_DL(gpu_ctx, P, d, vp))
    _close(ssd.laplace_SLDL(gpu_ctx, P, d, g, p, 0.5, 1.0), ssd.laplace_SLDL(gpu_ctx, P, d, g, vp, 0.5, 1.0))
    P.release()


@pytest.mark.parametrize("scale", [1.0, 1e-8, 1e-14, 1e-100])
def test_single_layer_beside_a_constant(gpu_ctx, scale):
    import torch

    import paper_2110_10749_gb300 as ssd
    q, const, _, f = _data(gpu_ctx, 1 / 8, scale)
    d = 3 / 8
    P = ssd.Points(q["xyz"], q["nrm"], q["w"]).prepare(gpu_ctx)
    _close(ssd.stokes_SLDL(gpu_ctx, P, d, 1.3, f, const, 0.5, -1.1), 0.5 * ssd.stokes_SL(gpu_ctx, P, d, 1.3, f))
    g, c = f[0].contiguous(), const[0].contiguous()
    _close(ssd.laplace_SLDL(gpu_ctx, P, d, g, c, 0.5, -1.1), 0.5 * ssd.laplace_SL(gpu_ctx, P, d, g))
    assert not ssd.stokes_DL(gpu_ctx, P, d, const).any() and not ssd.laplace_DL(gpu_ctx, P, d, c).any()
    # the first point has another value than the rest: nothing to subtract
    const[0, 0] = 2.0
    a = ssd.stokes_DL(gpu_ctx, P, d, const)
    const -= 1.0
    _close(a, ssd.stokes_DL(gpu_ctx, P, d, const))
    assert torch.isfinite(a).all()
    P.release()


def test_batch_of_constants_and_variations(gpu_ctx):
    import torch

    import paper_2110_10749_gb300 as ssd
    parts = [_data(gpu_ctx, h, s) for h, s in ((1 / 6, 1e-6), (1 / 5, 1.0), (1 / 8, 1e-9))]
    cat = lambda k: torch.cat([q[k] for q, *_ in parts], dim=-1).contiguous()
    n = [q["w"].numel() for q, *_ in parts]
    offs = np.concatenate([[0], np.cumsum(n)])
    delta = [3 / 6, 3 / 5, 3 / 8]
    B = ssd.Batch(cat("xyz"), cat("nrm"), cat("w"), offs, delta).prepare(gpu_ctx)
    u = torch.cat([c * (k + 1) + v for k, (_, c, v, _) in enumerate(parts)], dim=1)
    f = torch.cat([a for *_, a in parts], dim=1)
    rhs = lambda a: torch.stack([a, -2.0 * a]).contiguous()      # two right-hand sides
    out = ssd.batch_apply(gpu_ctx, B, ssd.OP_STOKES_DL, rhs(u))
    const = torch.cat([c * (k + 1) for k, (_, c, _, _) in enumerate(parts)], dim=1)
    fused = ssd.batch_apply(gpu_ctx, B, ssd.OP_STOKES_SLDL, rhs(const), rhs(f), mu=1.3, alpha=0.5, beta=1.0)
    for k, (q, _, v, a) in enumerate(parts):
        P = ssd.Points(q["xyz"], q["nrm"], q["w"])
        ref, single = ssd.stokes_DL(gpu_ctx, P, delta[k], v.contiguous()), ssd.stokes_SL(gpu_ctx, P, delta[k], 1.3, a)
        for r, s in ((0, 1.0), (1, -2.0)):
            _close(out[r][:, offs[k]:offs[k + 1]], s * ref)
            _close(fused[r][:, offs[k]:offs[k + 1]], s * 0.5 * single)
    B.release()


def test_a_plan_of_far_blocks(gpu_ctx):
    """Eight unit spheres on the corners of a cube: most block pairs are far, in launches of their own."""
    import torch

    import paper_2110_10749_gb300 as ssd
    q, const, var, _ = _data(gpu_ctx, 1 / 8, 1e-6)
    x = torch.cat([q["xyz"] + torch.tensor([[12.0 * (i >> 2 & 1)], [12.0 * (i >> 1 & 1)], [12.0 * (i & 1)]],
                                           dtype=torch.float64, device="cuda") for i in range(8)], dim=1).contiguous()
    P = ssd.Points(x, q["nrm"].repeat(1, 8), q["w"].repeat(8)).prepare(gpu_ctx)
    v = (var.repeat(1, 8) * torch.linspace(0.5, 1.0, 8, dtype=torch.float64, device="cuda").repeat_interleave(var.shape[1]))
    v[0] = _round(v[0])
    u = (const.repeat(1, 8) + v).contiguous()
    _close(ssd.stokes_DL(gpu_ctx, P, 3 / 8, u), ssd.stokes_DL(gpu_ctx, P, 3 / 8, v))
    before = gpu_ctx.launch_count()
    ssd.stokes_DL(gpu_ctx, P, 3 / 8, u)
    assert gpu_ctx.launch_count() - before == 4      # packing, near items, far items, epilogue
    P.release()
