"""The MALA step in one launch (proposals, set-up, likelihood and accept step in
the likelihood kernel) against the step in three (taken while trace events are
set): the same bits, for batches at the edges of the launch rule, chains outside
the prior box, next to its edges, unphysical ones, and draws u = 0 and 1."""
import numpy as np
import pytest

import synth
from tests._events import small_event

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sites", [("H1",), ("H1", "L1"), ("H1", "L1", "V1")])
def test_one_launch_equals_three(sites):
    import torch
    import paper_2404_11397_gb300 as rb
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    ev = small_event(sites=sites)
    event = rb.Event.from_synth(ev, n_bins=70)
    c = np.array(ev["theta_inj"], dtype=np.float64)
    c[9], c[12] = np.cos(c[9]), np.sin(c[12])
    half = np.array([0.01, 0.05, 0.02, 0.02, 250.0, 250.0, 20.0, 0.05, 0.5, 0.05, 0.5, 0.5, 0.2])
    lo, hi = c - half, c + half
    lo[9], hi[9], lo[12], hi[12] = max(lo[9], -1.0), min(hi[9], 1.0), max(lo[12], -1.0), min(hi[12], 1.0)
    rng = np.random.Generator(np.random.Philox(5))
    before, after = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    before.record(), after.record()
    for W in sorted({1, 3, 4, 5, 32, 33, 4 * n_sm - 1, 4 * n_sm + 1, 16 * n_sm + 1, 32 * n_sm - 1, 32 * n_sm, 32 * n_sm + 1}):
        z0 = lo + (hi - lo) * rng.uniform(0.0, 1.0, (W, 13))
        z0[W // 2, 9] = np.nextafter(hi[9], 0.0)      # next to the box's edge
        z0[W // 3, 1] = 1.5                           # outside it, and unphysical
        xi = rng.standard_normal((W, 13))
        xi[W // 4, 12] = 1e6                          # proposed far outside
        u = 1.0 - rng.random(W)
        u[0], u[-1] = (0.0, 1.0) if W > 1 else (0.5, 0.5)
        eps = 4e-4 * half
        out = []
        for traced in (False, True):
            try:
                rb.set_trace_events(before, after) if traced else rb.set_trace_events(None, None)
                z = torch.tensor(z0, device="cuda")
                logp, gz = rb.mala_init(event, z, lo, hi)
                first = [logp.clone(), gz.clone()]
                acc = [rb.mala_step(event, z, logp, gz, eps, lo, hi, torch.tensor(s * xi, device="cuda"),
                                    torch.tensor(u, device="cuda")) for s in (1.0, -1.0)]
                torch.cuda.synchronize()
            finally:
                rb.set_trace_events(None, None)
            out.append([t.cpu().numpy() for t in (*first, z, logp, gz, *acc)])
        for a, b in zip(*out):
            np.testing.assert_array_equal(a, b)
        if W > 100:
            assert 0 < out[0][-1].sum() < W
    event.free()
