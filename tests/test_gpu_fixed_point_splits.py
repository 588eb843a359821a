"""The FP64 operators on sets whose CTAs of 256 targets take chunks of sources
that are not whole blocks of 32 (a tile then touches up to five bounding
boxes): against the oracle's dense matrices, 1e-12 relative as for every FP64
operator."""
import numpy as np
import pytest

from oracle import quadrature as Q
from test_gpu_fixed_point import close, dense, device, subset

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1500, 2305, 2500])
@pytest.mark.parametrize("d", [0.4, 0.02])   # every pair smoothed; extent 100 delta, boxes that set a lower bound
def test_chunks_of_whole_ctas(gpu_ctx, n, d):
    import paper_2110_10749_gb300 as ssd
    p = subset(Q.ellipsoid_points((1.0, 0.7, 0.5), 1 / 18), n)
    rng = np.random.default_rng(n)
    dens = rng.normal(size=n), rng.normal(size=(3, n)), rng.normal(size=n), rng.normal(size=(3, n))
    P = ssd.Points.from_numpy(p).prepare(gpu_ctx)
    close(device(ssd, gpu_ctx, P, d, *dens), dense(p, d, *dens))
    P.release()
