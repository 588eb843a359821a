"""Off-surface fields on prepared points without a workspace of their own: a first call
under stream capture, where nothing may be allocated, and so many field points that
every block holds all sources and writes the result itself.  Tolerance 1e-12 against
the kernel in double precision (plain points)."""
import pytest

pytestmark = pytest.mark.gpu


def _calls(ssd, ctx, P, x, y):
    import torch
    f, u = torch.cos(3.0 * x).contiguous(), torch.sin(2.0 * x).contiguous()
    g, p = f[0].contiguous(), u[0].contiguous()
    return (lambda out: ssd.stokes_velocity_field(ctx, P, 1.3, (0.1, -0.2, 1.0), f, u, y, out=out),
            lambda out: ssd.darcy_pressure_field(ctx, P, 1.3, 0.4, g, p, y, out=out))


def _shell(q, nt):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(5)
    v = torch.randn(3, nt, dtype=torch.float64, device="cuda", generator=gen)
    return (v / v.norm(dim=0) * (1.5 + torch.rand(nt, dtype=torch.float64, device="cuda", generator=gen))).contiguous()


@pytest.mark.parametrize("which", [0, 1])
def test_first_call_under_capture(gpu_ctx, which):
    import torch

    import paper_2110_10749_gb300 as ssd
    q = ssd.quadrature_points(gpu_ctx, ssd.SPHERE, (1.0,), 1.0 / 8)
    y = _shell(q, 5000)
    ref = torch.empty((3, 5000) if which == 0 else 5000, dtype=torch.float64, device="cuda")
    _calls(ssd, gpu_ctx, ssd.Points(q["xyz"], q["nrm"], q["w"]), q["xyz"], y)[which](ref)
    cold = ssd.Context(0)
    P = ssd.Points(q["xyz"], q["nrm"], q["w"]).prepare(cold)
    call, out = _calls(ssd, cold, P, q["xyz"], y)[which], torch.empty_like(ref)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        for _ in range(2):   # cold, then with the pool that a plain call left
            graph = torch.cuda.CUDAGraph()
            graph.capture_begin()
            call(out)
            graph.capture_end()
            out.zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert float((out - ref).norm()) <= 1e-12 * float(ref.norm())
            call(out)
            torch.cuda.synchronize()
            assert float((out - ref).norm()) <= 1e-12 * float(ref.norm())
    P.release()
    cold.close()


@pytest.mark.parametrize("which", [0, 1])
def test_one_split(gpu_ctx, which):
    import torch

    import paper_2110_10749_gb300 as ssd
    q = ssd.quadrature_points(gpu_ctx, ssd.SPHERE, (1.0,), 1.0 / 4)
    nt = 256 * 16 * torch.cuda.get_device_properties(0).multi_processor_count + 5
    y = _shell(q, nt)
    out = [torch.empty((3, nt) if which == 0 else nt, dtype=torch.float64, device="cuda") for _ in range(2)]
    P = ssd.Points(q["xyz"], q["nrm"], q["w"])
    _calls(ssd, gpu_ctx, P, q["xyz"], y)[which](out[0])
    P.prepare(gpu_ctx)
    before = gpu_ctx.launch_count()
    _calls(ssd, gpu_ctx, P, q["xyz"], y)[which](out[1])
    assert gpu_ctx.launch_count() - before == 2      # packing and sums, no further pass over them
    assert float((out[1] - out[0]).norm()) <= 1e-12 * float(out[0].norm())
    P.release()
