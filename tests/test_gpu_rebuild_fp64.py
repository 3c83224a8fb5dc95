"""FP64 rebuild with a new theta_ref (h0 from FP64 Taylor chunks) against the
oracle's summary data: grids at the edge of the expansion's range (k_min =
1024, where the chunks are widest, and just below it, where the direct
evaluation runs), ragged grids (a partial last chunk), bins of one point, and
1, 2 and 3 detectors.

Tolerance: both sides evaluate phases of up to ~1e4 rad in FP64, so a point's term is
good to ~1e4 x a few 2^-52 ~ 1e-11, and the sums to less; 1e-9 of a
detector's largest entry, as the other FP64 builds are held to."""
import numpy as np
import pytest

import oracle
import synth
from tests._events import inject

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sites", [("H1",), ("H1", "L1"), ("H1", "L1", "V1")])
@pytest.mark.parametrize("T,f_low,f_high,n_bins", [
    (51.2, 20.0, 100.0, 37),      # k_min = 1024
    (51.15, 20.0, 100.0, 37),     # k_min = 1023: not expanded
    (64.0, 20.0, 512.3, 60),      # N not a multiple of the chunk
    (52.0, 20.0, 2048.0, 300),    # 1 / T not a power of two, parts of several chunks
    (64.0, 20.0, 21.5, 95),       # bins of one point, parts shorter than a chunk
])
def test_new_reference_rebuild_matches_oracle(sites, T, f_low, f_high, n_bins):
    import paper_2404_11397_gb300 as rb
    ev = inject(synth.make_event("C2", T=T, f_low=f_low, f_high=f_high, sites=sites))
    edges = oracle.bin_edges(ev, n_bins)
    event = rb.Event.from_synth(ev, n_bins=n_bins)
    ref = synth.posterior_box(ev["theta_inj"], 1, seed=311)[0]
    s = oracle.summary(ev, ref, edges)
    for kw in (dict(theta_ref=ref), dict()):  # generated, then streamed from the stored h0
        event.rebuild(mode="fp64", **kw)
        got = event.summary()
        for key in ("A0", "A1", "B0", "B1"):
            scale = np.max(np.abs(s[key]), axis=1, keepdims=True)
            assert np.max(np.abs(got[key] - s[key]) / scale) <= 1e-9, (key, kw)
    full = oracle.loglike_full(ev, ref)[0]
    assert abs(event.info()["base_logl"] - full) <= 1e-9 * np.sum(np.abs(s["B0"]) + np.abs(s["A0"]))
    event.free()
