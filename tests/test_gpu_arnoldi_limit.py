"""Local Stokes solves on either side of the longest vector of the one-launch Arnoldi
step (155648 entries): 51882 points run it, 51883 the separate kernels, which the
launches per step show.  The residual, formed with the FP64 operators, is within
twice the tolerance of the solve."""
import pytest

pytestmark = pytest.mark.gpu

TOL = 1e-9


def test_solves_around_the_longest_vector(gpu_ctx):
    import torch

    import paper_2110_10749_gb300 as ssd
    q = ssd.quadrature_points(gpu_ctx, ssd.SPHERE, (1.0,), 1.0 / 56)
    d, uinf = 3.0 / 56, (0.3, -0.2, 1.0)
    per_step, its = [], []
    for n in (51882, 51883):
        x, nrm, w = (q[k][..., :n].contiguous() for k in ("xyz", "nrm", "w"))
        f = torch.sin(2.0 * x).contiguous()
        P = ssd.Points(x, nrm, w).prepare(gpu_ctx)
        ssd.stokes_DL(gpu_ctx, P, d, f)              # the plan is made here
        before = gpu_ctx.launch_count()
        u, it, rel = ssd.stokes_solve(gpu_ctx, P, d, 1.0, f, uinf, ssd.krylov(TOL, 200, 60, False, ssd.FP64, True))
        per_step.append((gpu_ctx.launch_count() - before) / it)
        its.append(it)
        assert rel <= TOL
        b = torch.tensor(uinf, dtype=torch.float64, device="cuda")[:, None] - ssd.stokes_SL(gpu_ctx, P, d, 1.0, f)
        r = b - (u - ssd.stokes_DL(gpu_ctx, P, d, u) + nrm * ((u * nrm).sum(0) * w).sum() / w.sum())
        assert float(r.norm()) <= 2 * TOL * float(b.norm())
        P.release()
    assert abs(its[0] - its[1]) <= 1
    assert per_step[0] + 5 < per_step[1], per_step
