"""The two launch rules of mixed batches that the other batch-size tests stop short of:
gradient batches whose set-up takes its denser variant (more than 64 to 96 walkers per SM,
a wave fewer), against the same walkers in batches of one launch, and bin counts next
to an event's limit, where the tables leave no room for the walkers' records and a
small batch takes two kernels, against the two kernels of traced calls: bit for bit."""
import pytest

import synth
from tests._events import small_event

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sites", [("H1",), ("H1", "L1"), ("H1", "L1", "V1")])
def test_dense_setup_gives_the_rows_of_small_batches(sites):
    import torch
    import paper_2404_11397_gb300 as rb
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    event = rb.Event.from_synth(small_event(sites=sites), n_bins=70)
    sizes = (64 * n_sm, 64 * n_sm + 1, 80 * n_sm + 7, 96 * n_sm, 96 * n_sm + 1, 128 * n_sm + 33)
    theta = torch.tensor(synth.draw_prior(synth.PRIOR_GW170817, max(sizes), 78), device="cuda")
    theta[2, 1] = 1.5  # an unphysical walker among them
    small = [rb.loglike_grad(event, t) for t in theta.split(16 * n_sm)]
    L, G = (torch.cat(x) for x in zip(*small))
    for W in sizes:
        for at in (0, max(sizes) - W):
            l, g = rb.loglike_grad(event, theta[at:at + W])
            assert torch.equal(l, L[at:at + W]) and torch.equal(g, G[at:at + W]), (W, at)
    event.free()


@pytest.mark.parametrize("sites", [("H1",), ("H1", "L1", "V1")])
def test_bins_next_to_the_limit(sites):
    import torch
    import paper_2404_11397_gb300 as rb
    ev = small_event(sites=sites)
    before, after = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    before.record(), after.record()
    theta = torch.tensor(synth.posterior_box(ev["theta_inj"], 70, seed=6), device="cuda")
    launches = []
    lo, hi = 500, ev["N"] - 1  # the largest admitted bin count, then steps of a slot group's bins below it
    while hi - lo > 1:
        mid = (lo + hi) // 2
        try:
            rb.Event.from_synth(ev, n_bins=mid).free()
            lo = mid
        except rb.RBError:
            hi = mid
    for n_bins in (lo - 4 * 62, lo - 3 * 62, lo - 2 * 62, lo - 62, lo):
        event = rb.Event.from_synth(ev, n_bins=n_bins)
        n0 = rb.kernel_launch_count()
        got = [*rb.loglike_grad(event, theta), rb.loglike(event, theta)]
        launches.append(rb.kernel_launch_count() - n0)
        rb.set_trace_events(before, after)
        try:
            ref = [*rb.loglike_grad(event, theta), rb.loglike(event, theta)]
            torch.cuda.synchronize()
        finally:
            rb.set_trace_events(None, None)
        for a, b in zip(got, ref):
            assert torch.equal(a, b), n_bins
        assert torch.isfinite(got[0]).all()
        event.free()
    assert launches[0] == 2 and launches[-1] == 4, launches
