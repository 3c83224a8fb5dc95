"""Workspace of a large full-grid batch: what include/rb.h says of it (176 B per walker
and 64 MiB), seen as the device memory taken while the call's kernels still run, and
walkers beyond the first tile (21 840 on a grid of 64 groups) get the bits that they
get alone."""
import numpy as np
import pytest
import torch

import synth
from tests.test_gpu_full import Case, rb  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu


def test_workspace_of_a_large_batch_is_bounded(rb):  # noqa: F811
    c = Case(rb, "C2", n_bins=2, T=64.0, f_low=20.0, f_high=20.0 + (64 * 2048 - 1) / 64.0, sites=("H1",))
    few = torch.tensor(synth.posterior_box(c.ev["theta_inj"], 100, seed=3), device="cuda")
    W = 600_000
    theta = few.repeat(W // 100, 1)
    ref = rb.loglike_full(c.event, few)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    L = rb.loglike_full(c.event, theta)
    taken = before - torch.cuda.mem_get_info()[0]
    torch.cuda.synchronize()
    # L itself and the pool's rounding to 32 MiB pieces beside it
    assert taken <= 176 * W + (64 << 20) + 8 * W + (64 << 20)
    assert torch.equal(L.view(-1, 100), ref.expand(W // 100, 100))
    assert np.isfinite(ref.cpu().numpy()).all()
    c.event.free()
