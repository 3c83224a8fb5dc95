"""Full-grid likelihood at the edges of its kernel's tiling: grids of a few
points, one chunk (32 points) and one segment (64 chunks) more or less, ragged
last chunks, and batches around a block's eight walkers, for 1, 2 and 3
detectors, against the oracle with test_gpu_full's tolerance (derived there);
every batch gives a walker the same bits."""
import numpy as np
import pytest
import torch

import synth
from tests.test_gpu_full import Case, rb  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sites", [("H1",), ("H1", "L1"), ("H1", "L1", "V1")])
@pytest.mark.parametrize("points", [3, 31, 32, 33, 1024, 1025, 2047, 2048, 2049, 64 * 2048 + 40])
def test_grid_and_batch_edges(rb, sites, points):  # noqa: F811
    T, f_low = 64.0, 20.0
    if len(sites) > 1 and points > 100000:
        T = 72.0
    c = Case(rb, "C2", n_bins=2, T=T, f_low=f_low, f_high=f_low + (points - 1) / T, sites=sites)
    assert c.ev["N"] == points
    theta = synth.posterior_box(c.ev["theta_inj"], 17, seed=points)
    whole, _ = c.check(rb, theta)
    for a, b in ((0, 1), (3, 4), (0, 7), (1, 9), (4, 12), (0, 9)):
        part = rb.loglike_full(c.event, torch.tensor(theta[a:b], device="cuda")).cpu().numpy()
        np.testing.assert_array_equal(part, whole[a:b])
    c.event.free()
