"""Local solves on the one-launch Arnoldi step: lengths around its blocks of 64
rows, one block, restarts after a few steps and many vectors in one cycle,
against dense solves of the oracle's matrices.  Solves to a relative residual
of 1e-12 of systems with condition numbers below 1e3: 1e-9 in the solution."""
import numpy as np
import pytest

import oracle
from oracle import quadrature as Q

pytestmark = pytest.mark.gpu

H = 1 / 6


@pytest.fixture(scope="module")
def cloud():
    return Q.ellipsoid_points((1.0, 0.8, 0.6), H)


def check(out, ref):
    assert np.linalg.norm(out - ref) <= 1e-9 * np.linalg.norm(ref)


@pytest.mark.parametrize("n", [7, 63, 64, 65, 129, 321])
@pytest.mark.parametrize("restart", [4, 80])
def test_darcy_solves_match_dense_solves(gpu_ctx, cloud, n, restart):
    # -D^L p + (w . p) / W = (mu/kappa) L q, zero weighted mean
    import torch
    import paper_2110_10749_gb300 as ssd
    k = np.linspace(0, cloud["w"].size - 1, n).astype(int)
    p = {q: np.ascontiguousarray(cloud[q][..., k]) for q in ("xyz", "nrm", "w")}
    p["w"] = p["w"] * (cloud["w"].sum() / p["w"].sum())
    d, W = 3 * H, p["w"].sum()
    q = np.random.default_rng(n).normal(size=n)
    P = ssd.Points.from_numpy(p).prepare(gpu_ctx)
    kr = ssd.krylov(1e-12, 400, restart, False, ssd.FP64)
    sol, its, rel = ssd.darcy_solve(gpu_ctx, P, d, 1.3, 0.4, torch.as_tensor(q, device="cuda"), kr)
    P.release()
    A = -oracle.operator_matrix(p, d, "DL") + np.outer(np.ones(n), p["w"]) / W
    ref = np.linalg.solve(A, 1.3 / 0.4 * oracle.operator_matrix(p, d, "L") @ q)
    assert rel <= 1e-12
    check(sol.cpu().numpy(), ref - (p["w"] @ ref) / W)


@pytest.mark.parametrize("h", [1 / 3, 1 / 5, 1 / 6])
@pytest.mark.parametrize("restart", [20, 80])   # GMRES(12) stagnates on h = 1/5 (scipy's too)
def test_stokes_solves_match_dense_solves(gpu_ctx, h, restart):
    # (I - D^S) u + n (w . (u . n)) / W = U - M f, whole quadrature sets
    import torch
    import paper_2110_10749_gb300 as ssd
    p = Q.ellipsoid_points((1.0, 0.8, 0.6), h)
    n, d, W = p["w"].size, 3 * h, p["w"].sum()
    f = np.random.default_rng(n).normal(size=(3, n))
    P = ssd.Points.from_numpy(p).prepare(gpu_ctx)
    kr = ssd.krylov(1e-12, 400, restart, False, ssd.FP64, deflate=True)
    sol, its, rel = ssd.stokes_solve(gpu_ctx, P, d, 1.0, torch.as_tensor(f, device="cuda"), (0.3, -0.2, 1.0), kr)
    P.release()
    nv = p["nrm"].reshape(-1)
    B = np.eye(3 * n) - oracle.operator_matrix(p, d, "DS") + np.outer(nv, (p["nrm"] * p["w"]).reshape(-1)) / W
    ref = np.linalg.solve(B, np.repeat([0.3, -0.2, 1.0], n) - oracle.operator_matrix(p, d, "M") @ f.reshape(-1))
    assert rel <= 1e-12
    check(sol.cpu().numpy().reshape(-1), ref)
