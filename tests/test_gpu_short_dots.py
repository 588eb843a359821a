"""Dot products around the lengths where one launch takes over from two, by the
contraction of point derivatives (25 coefficients, vectors of 3n, 3n and n).
A sum of m products in any order is within m 2^-53 of the sum of magnitudes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 170, 171, 511, 513, 2730, 2731, 8192, 8193])
def test_contraction_at_short_lengths(gpu_ctx, n):
    import torch

    import paper_2110_10749_gb300 as ssd
    rng = np.random.default_rng(n)
    jac = {"dxyz": rng.normal(size=(25, 3, n)), "dnrm": rng.normal(size=(25, 3, n)), "dw": rng.normal(size=(25, n))}
    geo = [rng.normal(size=(3, n)), rng.normal(size=(3, n)), rng.normal(size=n)]
    out = ssd.shape_contract(gpu_ctx, {k: torch.as_tensor(v, device="cuda") for k, v in jac.items()},
                             [torch.as_tensor(v, device="cuda") for v in geo])
    out = np.asarray(out.cpu() if hasattr(out, "cpu") else out)
    ref, mag = np.zeros(25), np.zeros(25)
    for J, g in zip((jac["dxyz"], jac["dnrm"], jac["dw"]), geo):
        t = J.reshape(25, -1) * g.reshape(1, -1)
        ref += t.astype(np.longdouble).sum(axis=1).astype(float)
        mag += np.abs(t).sum(axis=1)
    assert (np.abs(out - ref) <= (7 * n + 4) * 2.0 ** -53 * mag).all()
