"""The geometric derivative sums at the sizes where the split of the partners
over a CTA of 128 threads has edges."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MU = 1.3


def _bilinear(torch, name, x, nr, w, d, a, b):
    """a . (K b) from the closed forms of the smoothing factors."""
    n = w.shape[0]
    off = ~torch.eye(n, dtype=torch.bool)
    D = x[:, :, None] - x[:, None, :]
    r2 = torch.where(off, (D * D).sum(0), torch.ones((), dtype=x.dtype))
    r = r2.sqrt()
    t = r2 / d ** 2
    E = torch.exp(-t) * 2 / math.sqrt(math.pi) * r / d
    er = torch.erf(r / d)
    s1 = er - E * (2 * t - 5) / 3
    s2 = er + E * (2 * t - 3) / 3
    s3 = er - E * (4 * t * t - 14 * t + 3) / 3
    s4 = er - E * (8 * t ** 3 - 36 * t * t + 6 * t + 9) / 9
    c1 = 16 / (3 * math.sqrt(math.pi)) / d
    m = off.to(x.dtype)
    if name == "LSL":
        return -(((a[:, None] * b[None] * s1 / r * m) * w).sum() + c1 * (a * b * w).sum()) / (4 * math.pi)
    if name == "LDL":
        dn = (D * nr[:, None, :]).sum(0)
        return -(a[:, None] * (b[None] - b[:, None]) * w * dn * s2 / r ** 3 * m).sum() / (4 * math.pi)
    aD = (a[:, :, None] * D).sum(0)
    if name == "SSL":
        ab = (a[:, :, None] * b[:, None, :]).sum(0)
        bD = (b[:, None, :] * D).sum(0)
        pair = ((s1 / r * ab + s3 / r ** 3 * aD * bD) * m * w).sum()
        return (pair + c1 * ((a * b).sum(0) * w).sum()) / (8 * math.pi * MU)
    bD = ((b[:, None, :] - b[:, :, None]) * D).sum(0)
    dn = (D * nr[:, None, :]).sum(0)
    return 6 / (8 * math.pi) * (w * s4 / r ** 5 * aD * bD * dn * m).sum()


@pytest.mark.parametrize("n", [1, 2, 127, 128, 129, 257])
@pytest.mark.parametrize("name", ["LSL", "LDL", "SSL", "SDL"])
def test_geometry_gradient_sizes(gpu_ctx, name, n):
    import torch

    import paper_2110_10749_gb300 as ssd
    # a Fibonacci sphere keeps r / delta above 0.9, where the closed forms lose
    # less than 1e3 ulp, and reaches past 8 delta; 257 terms a point: 1e-11 of
    # the largest entry is a factor 10 above both
    i = np.arange(n) + 0.5
    z = 1 - 2 * i / n
    ph = i * math.pi * (3 - math.sqrt(5))
    s = np.sqrt(1 - z * z)
    rng = np.random.default_rng(n)
    x = np.stack([s * np.cos(ph), s * np.sin(ph), z])
    nrm = x + 0.1 * rng.normal(size=(3, n))
    w = rng.uniform(0.5, 1.5, size=n)
    nc = (3, n) if name[0] == "S" else n
    a, b = rng.normal(size=nc), rng.normal(size=nc)
    d = 0.2
    tx, tn, tw = (torch.tensor(v, requires_grad=True) for v in (x, nrm, w))
    _bilinear(torch, name, tx, tn, tw, d, torch.tensor(a), torch.tensor(b)).backward()
    ref = [np.zeros_like(v.detach().numpy()) if v.grad is None else v.grad.numpy() for v in (tx, tn, tw)]
    dev = [torch.as_tensor(v, device="cuda") for v in (x, nrm, w)]
    op = {"LSL": ssd.OP_LAPLACE_SL, "LDL": ssd.OP_LAPLACE_DL, "SSL": ssd.OP_STOKES_SL, "SDL": ssd.OP_STOKES_DL}[name]
    got = ssd.geometry_gradient(gpu_ctx, ssd.Points(*dev), op, d, torch.as_tensor(a, device="cuda"),
                                torch.as_tensor(b, device="cuda"), mu=MU)
    for g, r in zip(got, ref):
        assert np.abs(g.cpu().numpy() - r).max() <= 1e-11 * max(np.abs(r).max(), 1e-300)
