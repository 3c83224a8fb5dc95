"""log L(theta_ref) of an FP64 build that generates its fiducial waveform is the FP64
sum of the bins' shares Re A0 - B0 / 2: against their exact sum.  Tolerance: at most 4096
shares, each addition of the pairwise sums within 2^-53 of a partial sum, ~32 additions
on the way of a share, and the share's own rounding: 2^-53 (32 + 1) < 4e-15 of the sum of
moduli."""
import math

import numpy as np
import pytest

import synth
from tests._events import inject

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sites", [("H1",), ("H1", "L1"), ("H1", "L1", "V1")])
@pytest.mark.parametrize("T,n_bins", [(64.0, 1), (64.0, 700), (51.15, 300)])
def test_base_is_the_fp64_sum_of_the_shares(sites, T, n_bins):
    import paper_2404_11397_gb300 as rb
    ev = inject(synth.make_event("C2", T=T, f_high=500.0, sites=sites))
    event = rb.Event.from_synth(ev, n_bins=n_bins)
    for ref in (None, synth.posterior_box(ev["theta_inj"], 1, seed=9)[0]):
        if ref is not None:
            event.rebuild(theta_ref=ref, mode="fp64")
        s = event.summary()
        shares = (s["A0"].real - 0.5 * s["B0"]).ravel()
        assert abs(event.info()["base_logl"] - math.fsum(shares)) <= 4e-15 * np.sum(np.abs(shares))
    event.free()
