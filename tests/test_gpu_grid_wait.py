"""The bounded waits of the one-launch Arnoldi step: with no poll allowed every
block gives up at its first barrier, and the solve says so with a status of its own
(not the one of data that is not finite) and leaves the device usable."""
import pytest

pytestmark = pytest.mark.gpu


def _solve(ssd, ctx, P, u):
    kr = ssd.krylov(1e-10, 200, 50, False, ssd.FP64)
    return ssd.stokes_solve(ctx, P, 3.0 / 8, 1.0, u, (0.3, -0.2, 1.0), kr)[0]


def test_a_wait_that_runs_out_is_reported(gpu_ctx, monkeypatch):
    import torch

    import paper_2110_10749_gb300 as ssd
    q = ssd.quadrature_points(gpu_ctx, ssd.SPHERE, (1.0,), 1.0 / 8)
    u = torch.sin(2.0 * q["xyz"]).contiguous()
    P = ssd.Points(q["xyz"], q["nrm"], q["w"]).prepare(gpu_ctx)
    expect = _solve(ssd, gpu_ctx, P, u)
    monkeypatch.setenv("SSD_GRID_POLLS", "0")
    short = ssd.Context(0)
    monkeypatch.delenv("SSD_GRID_POLLS")
    R = ssd.Points(q["xyz"], q["nrm"], q["w"]).prepare(short)
    for _ in range(2):   # the frame is used again
        with pytest.raises(ssd.SsdError, match="grid barrier") as e:
            _solve(ssd, short, R, u)
        assert e.value.status == ssd.SSD_ECUDA
    short.sync()
    R.release()
    short.close()
    assert torch.equal(_solve(ssd, gpu_ctx, P, u), expect)
    u[1, 5] = float("nan")
    with pytest.raises(ssd.SsdError) as e:
        _solve(ssd, gpu_ctx, P, u)
    assert e.value.status == ssd.SSD_ENUMERIC
    P.release()
