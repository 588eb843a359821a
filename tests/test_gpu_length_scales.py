"""Lengths at the ends of what the arithmetic holds.  Single precision: at delta =
1.5e-19 the squared distances of close pairs are subnormal (delta^2 / 4 to 1.2e-38).
The Laplace single layer needs no higher power of 1 / delta, so it stays in range;
tolerance 1e-5 against FP64, as for every FP32C operator.  Double precision: off-surface
fields scale with the length by exact powers, 1e-12 at every one."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("delta", [1e-19, 1.5e-19, 2.1e-19, 2.3e-19])
@pytest.mark.parametrize("prepared", [False, True])
def test_laplace_single_layer_with_subnormal_squared_distances(gpu_ctx, delta, prepared):
    import numpy as np
    import torch

    import paper_2110_10749_gb300 as ssd
    q = ssd.quadrature_points(gpu_ctx, ssd.SPHERE, (1.0,), 1.0 / 8)
    s = delta * 8 / 3
    x, w = (s * q["xyz"]).contiguous(), (s * s * q["w"]).contiguous()
    P = ssd.Points(x, q["nrm"], w)
    if prepared:
        P.prepare(gpu_ctx)
    g = torch.cos(3.0 * q["xyz"][0]).contiguous()
    ref = ssd.laplace_SL(gpu_ctx, P, delta, g)
    B = ssd.Batch(x, q["nrm"], w, np.array([0, w.numel()]), np.array([delta])).prepare(gpu_ctx)
    for out in (ssd.laplace_SL(gpu_ctx, P, delta, g, ssd.FP32C),
                ssd.batch_apply(gpu_ctx, B, ssd.OP_LAPLACE_SL, g[None], prec=ssd.FP32C).view(-1)):
        assert float((out - ref).norm()) <= 1e-5 * float(ref.norm())
    B.release()
    P.release()


@pytest.mark.parametrize("s", [1e-80, 1e-60, 1e60, 1e80])
@pytest.mark.parametrize("prepared", [False, True])
def test_off_surface_fields_scale_with_the_length(gpu_ctx, s, prepared):
    import torch

    import paper_2110_10749_gb300 as ssd
    q = ssd.quadrature_points(gpu_ctx, ssd.SPHERE, (1.0,), 1.0 / 6)
    x, w = q["xyz"], q["w"]
    y = (2.5 * x[:, ::3]).contiguous()
    f, u = torch.cos(3.0 * x).contiguous(), torch.sin(2.0 * x).contiguous()

    def fields(t):
        P = ssd.Points((t * x).contiguous(), q["nrm"], (t * t * w).contiguous())
        if prepared:
            P.prepare(gpu_ctx)
        ft, yt = (f / t).contiguous(), (t * y).contiguous()
        out = (ssd.stokes_velocity_field(gpu_ctx, P, 1.3, (0.1, 0.2, 1.0), ft, u, yt),
               ssd.darcy_pressure_field(gpu_ctx, P, 1.3, 0.4, ft[0].contiguous(), u[0].contiguous(), yt),
               t * ssd.stokes_pressure_field(gpu_ctx, P, 1.3, ft, u, yt))
        P.release()
        return out

    for a, b in zip(fields(s), fields(1.0)):
        assert float((a - b).norm()) <= 1e-12 * float(b.norm())


@pytest.mark.parametrize("s", [1e-110, 1e-105, 1e100])
def test_darcy_pressure_at_extreme_lengths(gpu_ctx, s):
    import torch

    import paper_2110_10749_gb300 as ssd
    q = ssd.quadrature_points(gpu_ctx, ssd.SPHERE, (1.0,), 1.0 / 6)
    x, w = q["xyz"], q["w"]
    g, p = torch.cos(3.0 * x[0]).contiguous(), torch.sin(2.0 * x[1]).contiguous()
    out = []
    for t in (s, 1.0):
        P = ssd.Points((t * x).contiguous(), q["nrm"], (t * t * w).contiguous())
        out.append(ssd.darcy_pressure_field(gpu_ctx, P, 1.3, 0.4, (g / t).contiguous(), p, (2.5 * t * x).contiguous()))
    assert float((out[0] - out[1]).norm()) <= 1e-12 * float(out[1].norm())
