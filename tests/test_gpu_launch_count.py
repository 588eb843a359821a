"""The launch counter counts the kernels that run: the bounding box of a prepared set is
one launch up to 4096 points and two beyond, with the rest of the layout the same."""
import pytest

pytestmark = pytest.mark.gpu


def test_preparing_small_and_large_sets(gpu_ctx):
    import numpy as np
    import torch

    import paper_2110_10749_gb300 as ssd
    gen = torch.Generator(device="cuda").manual_seed(1)
    counts = {}
    for n in (500, 4096, 4097, 9000):
        x = torch.randn(3, n, dtype=torch.float64, device="cuda", generator=gen)
        nrm, w = (x / x.norm(dim=0)).contiguous(), torch.ones(n, dtype=torch.float64, device="cuda")
        for kind in ("points", "batch"):
            before = gpu_ctx.launch_count()
            P = (ssd.Points(x, nrm, w) if kind == "points" else
                 ssd.Batch(x, nrm, w, np.array([0, n]), np.array([0.5]))).prepare(gpu_ctx)
            counts[kind, n] = gpu_ctx.launch_count() - before
            P.release()
    for kind in ("points", "batch"):
        assert counts[kind, 500] == counts[kind, 4096]
        assert counts[kind, 4097] == counts[kind, 9000] == counts[kind, 500] + 1
