"""Off-surface fields on prepared point sets (fixed point) and plain ones
(double precision): field-point counts around the blocks, points that mix all
cases in one call (ordinary, closer than a point spacing, 40 extents out, not
finite), densities without a common scale.  Tolerance 1e-12 of the sums, as for
the representations' other tests."""
import numpy as np
import pytest

from oracle import field as F
from oracle import quadrature as Q

pytestmark = pytest.mark.gpu

KAPPA, MU, UINF = 0.3, 1.3, (0.2, -0.4, 1.0)


@pytest.fixture(scope="module")
def body(gpu_ctx):
    import paper_2110_10749_gb300 as ssd
    p = Q.ellipsoid_points((1.0, 0.7, 0.5), 1 / 10, center=(0.3, 0.0, -5.0))
    P, R = ssd.Points.from_numpy(p), ssd.Points.from_numpy(p).prepare(gpu_ctx)
    yield p, P, R
    R.release()


def shell(p, nt, seed):
    rng = np.random.default_rng(seed)
    v = rng.normal(size=(3, nt))
    return p["xyz"].mean(axis=1)[:, None] + v / np.linalg.norm(v, axis=0) * rng.uniform(1.3, 4.0, nt)


def both(gpu_ctx, body, y, q, pd, f, u, uinf=UINF):
    import torch
    import paper_2110_10749_gb300 as ssd
    p, P, R = body
    T = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    for pts in (P, R):
        yield (ssd.stokes_velocity_field(gpu_ctx, pts, MU, uinf, T(f), T(u), T(y)).cpu().numpy(),
               ssd.darcy_pressure_field(gpu_ctx, pts, MU, KAPPA, T(q), T(pd), T(y)).cpu().numpy(),
               ssd.stokes_pressure_field(gpu_ctx, pts, MU, T(f), T(u), T(y)).cpu().numpy())


def reference(p, y, q, pd, f, u, uinf=UINF):
    return (F.stokes_velocity_field(p, f, u, MU, uinf, y), F.darcy_pressure_field(p, q, pd, MU, KAPPA, y),
            F.stokes_pressure_field(p, f, u, MU, y))


def data(p, seed):
    rng = np.random.default_rng(seed)
    n = p["w"].size
    return rng.normal(size=n), rng.normal(size=n), rng.normal(size=(3, n)), rng.normal(size=(3, n))


@pytest.mark.parametrize("nt", [1, 63, 65, 255, 257, 4095, 4097])
def test_counts_around_the_blocks(gpu_ctx, body, nt):
    p = body[0]
    y, d = shell(p, nt, nt), data(p, 1)
    ref = reference(p, y, *d)
    for out in both(gpu_ctx, body, y, *d):
        for a, b in zip(out, ref):
            assert np.linalg.norm(a - b) <= 1e-12 * np.linalg.norm(b)


def test_all_kinds_of_field_points_in_one_call(gpu_ctx, body):
    p = body[0]
    y, d = shell(p, 400, 3), data(p, 2)
    near = p["xyz"][:, :60] + 1e-3 * p["nrm"][:, :60]          # closer than a point spacing (0.1)
    far = p["xyz"].mean(axis=1)[:, None] + 80.0 * np.eye(3)
    y[:, 10:70], y[:, 100:103] = near, far
    ref = reference(p, y, *d)
    for out in both(gpu_ctx, body, y, *d):
        for a, b in zip(out, ref):
            # every point on its own: the far ones are small, the near ones large
            err, mag = np.abs(a - b).reshape(-1, 400).max(axis=0), np.abs(b).reshape(-1, 400).max(axis=0)
            assert (err <= 1e-11 * (mag + np.median(mag) * 1e-3)).all()
    y[0, 5], y[2, 6] = np.nan, np.inf
    for out in both(gpu_ctx, body, y, *d):
        assert not np.isfinite(out[0][:, 5]).any() and np.isfinite(out[0][:, 7:]).all()
        assert np.isnan(out[1][5]) and np.isfinite(out[1][7:]).all()


@pytest.mark.parametrize("scale", [1e-90, 1e90, 1e200])
def test_density_scales(gpu_ctx, body, scale):
    # 1e200 is out of the fixed-point range: double precision inside the same launch
    p = body[0]
    y = shell(p, 130, 5)
    q, pd, f, u = data(p, 4)
    zero = (0.0, 0.0, 0.0)
    ref = reference(p, y, q, pd, f, u, zero)
    for out in both(gpu_ctx, body, y, scale * q, scale * pd, scale * f, scale * u, zero):
        for a, b in zip(out, ref):
            assert np.linalg.norm(a / scale - b) <= 1e-12 * np.linalg.norm(b)


def test_non_finite_densities(gpu_ctx, body):
    p = body[0]
    y = shell(p, 40, 6)
    q, pd, f, u = data(p, 5)
    q[3] = f[1, 3] = np.nan
    for out in both(gpu_ctx, body, y, q, pd, f, u):
        assert np.isnan(out[0]).all() and np.isnan(out[1]).all() and np.isnan(out[2]).all()
