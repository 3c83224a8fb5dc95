"""Full-grid likelihood where its phase sums have to work hardest or least: the
smallest admitted T f_low (1024: the high Taylor orders, terms of several turns per
step), bands above 150 Hz (those orders left out), a grid that has both, and
walkers far from the event in the masses, the tides and the time, against the
oracle with test_gpu_full's tolerance.  A walker whose phase coefficients are beyond
FP32 gives NaN, and nothing to the others."""
import numpy as np
import pytest
import torch

import synth
from tests.test_gpu_full import Case, rb  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,f_low,f_high", [(51.2, 20.0, 90.0), (64.0, 16.0, 500.0), (64.0, 150.0, 300.0), (128.0, 40.0, 400.0)])
@pytest.mark.parametrize("sites", [("H1",), ("H1", "L1", "V1")])
def test_phase_ranges(rb, sites, T, f_low, f_high):  # noqa: F811
    c = Case(rb, "C2", n_bins=2, T=T, f_low=f_low, f_high=f_high, sites=sites)
    theta = synth.posterior_box(c.ev["theta_inj"], 12, seed=3)
    theta[1, 0] *= 0.8
    theta[2, 0] *= 1.7
    theta[3, 1] = 0.2
    theta[4, 4:6] = 5000.0
    theta[5, 7] = 0.4
    theta[6, 7] = -0.4
    theta[7, 2:4] = -0.8, 0.9
    c.check(rb, theta)
    c.event.free()


def test_a_phase_out_of_range_is_not_a_number(rb):  # noqa: F811
    c = Case(rb, "C2", n_bins=2, T=64.0, f_low=20.0, f_high=200.0, sites=("H1",))
    theta = synth.posterior_box(c.ev["theta_inj"], 9, seed=4)
    ref = rb.loglike_full(c.event, torch.tensor(theta, device="cuda")).cpu().numpy()
    theta[3, 0] = 1e-26  # phase coefficients beyond FP32
    got = rb.loglike_full(c.event, torch.tensor(theta, device="cuda")).cpu().numpy()
    assert np.isnan(got[3])
    keep = np.arange(9) != 3
    np.testing.assert_array_equal(got[keep], ref[keep])
    c.event.free()
