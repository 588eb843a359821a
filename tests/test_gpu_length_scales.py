"""Lengths at the ends of what single precision holds: at delta = 1.5e-19 the squared
distances of close pairs are subnormal (delta^2 / 4 to 1.2e-38).  The Laplace single
layer needs no higher power of 1 / delta, so it stays in range; tolerance 1e-5
against FP64, as for every FP32C operator."""
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
