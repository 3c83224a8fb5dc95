"""Batch sizes at the edges of the likelihood kernel's launch rule (walkers
spread over the SMs, dense blocks, several rounds): a walker's result does not
depend on the batch it is in, so the rows of every size equal, bit for bit,
those of one large batch (which the parity tests compare with the oracle)."""
import numpy as np
import pytest

import synth
from tests._events import small_event

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sites", [("H1",), ("H1", "L1"), ("H1", "L1", "V1")])
@pytest.mark.parametrize("grad", [True, False])
@pytest.mark.parametrize("mode", ["mixed", "fp64"])
def test_results_do_not_depend_on_the_batch_size(sites, grad, mode):
    import torch
    import paper_2404_11397_gb300 as rb
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    event = rb.Event.from_synth(small_event(sites=sites), n_bins=70)
    sizes = sorted({1, 3, 4, 5, 31, 32, 33, 4 * n_sm - 1, 8 * n_sm, 8 * n_sm + 1, 4 * n_sm, 4 * n_sm + 1, 16 * n_sm - 1, 16 * n_sm, 16 * n_sm + 1,
                    32 * n_sm, 32 * n_sm + 1})
    W = 40 * n_sm + 7
    theta = torch.tensor(synth.draw_prior(synth.PRIOR_GW170817, W, 77), device="cuda")
    theta[2, 1] = 1.5  # an unphysical walker among them
    call = (lambda t: rb.loglike_grad(event, t, mode)) if grad else (lambda t: (rb.loglike(event, t, mode),))
    whole = [x.cpu().numpy() for x in call(theta)]
    for w in sizes:
        for part, ref in zip(call(theta[:w]), whole):
            assert np.array_equal(part.cpu().numpy(), ref[:w]), w
        # and from another offset: other lanes, warps and blocks
        for part, ref in zip(call(theta[W - w:]), whole):
            assert np.array_equal(part.cpu().numpy(), ref[W - w:]), w
    event.free()
