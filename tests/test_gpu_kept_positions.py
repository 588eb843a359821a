"""Grid positions that are kept with a layout for one smoothing radius: a replayed
graph, and a second context on the same layout, give what a plain call gives
(the same pairs in the same order: the same bits) whatever radii were used in between."""
import pytest

pytestmark = pytest.mark.gpu

RADII = (3.0 / 8, 4.0 / 8)


def _inputs(ctx):
    import torch

    import paper_2110_10749_gb300 as ssd
    q = ssd.quadrature_points(ctx, ssd.SPHERE, (1.0,), 1.0 / 8)
    u = torch.sin(2.0 * q["xyz"]).contiguous()
    return ssd.Points(q["xyz"], q["nrm"], q["w"]).prepare(ctx), u


def _calls(ssd, ctx, P, u):
    return {"stokes_DL": lambda d: ssd.stokes_DL(ctx, P, d, u, ssd.FP64),
            "stokes_SLDL": lambda d: ssd.stokes_SLDL(ctx, P, d, 1.3, u, u, 0.7, -1.1, ssd.FP64)}


@pytest.mark.parametrize("name", ["stokes_DL", "stokes_SLDL"])
def test_graph_replays_after_another_radius(gpu_ctx, name):
    import torch

    import paper_2110_10749_gb300 as ssd
    P, u = _inputs(gpu_ctx)
    call = _calls(ssd, gpu_ctx, P, u)[name]
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        other = call(RADII[1]).clone()
        expect = call(RADII[0]).clone()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        graph.capture_begin()
        out = call(RADII[0])
        graph.capture_end()
        assert torch.equal(call(RADII[0]), expect)      # before any replay
        assert torch.equal(call(RADII[1]), other)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, expect)
        assert torch.equal(call(RADII[1]), other)
        torch.cuda.synchronize()
    P.release()


def test_two_contexts_on_one_layout(gpu_ctx):
    import torch

    import paper_2110_10749_gb300 as ssd
    P, u = _inputs(gpu_ctx)
    second = ssd.Context(0)
    first, other = _calls(ssd, gpu_ctx, P, u), _calls(ssd, second, P, u)
    for name in first:
        expect = [first[name](d).clone() for d in RADII]
        for k in (0, 1, 0):
            assert torch.equal(other[name](RADII[k]), expect[k])
            assert torch.equal(first[name](RADII[1 - k]), expect[1 - k])
    torch.cuda.synchronize()
    P.release()
