"""The sampled quadrature where a line takes more than one window of 512
samples and the last CTA has fewer than its 8 lines."""
import numpy as np
import pytest

from oracle import quadrature as Q

pytestmark = pytest.mark.gpu


def test_wide_molecule_points_match_oracle(gpu_ctx):
    """Width 3: 640 samples a line, two windows; every label and coordinate equal."""
    import paper_2110_10749_gb300 as ssd
    g = {k: v.cpu().numpy() for k, v in ssd.molecule_points(gpu_ctx, 1 / 2, r=3.0).items()}
    o = Q.molecule_points(1 / 2, r=3.0)
    assert np.array_equal(g["meta"], o["meta"])
    assert np.array_equal(g["xyz"], o["xyz"])
    assert np.array_equal(g["nrm"], o["nrm"])
