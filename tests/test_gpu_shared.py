"""RB_SHARED: batches and MALA steps that share the GPU with others give the bits of the
default form, with as many kernels as the form with few, dense blocks has; calls that
have no such form refuse the flag."""
import numpy as np
import pytest

import synth
from tests._events import small_event

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sites", [("H1",), ("H1", "L1"), ("H1", "L1", "V1")])
@pytest.mark.parametrize("mode", ["mixed", "mixed_f64phase"])
def test_same_bits_as_the_default_form(sites, mode):
    import torch
    import paper_2404_11397_gb300 as rb
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    ev = small_event(sites=sites)
    event = rb.Event.from_synth(ev, n_bins=70)
    for W in (1, 5, 16, 17, 4 * n_sm + 1, 16 * n_sm + 1, 32 * n_sm, 32 * n_sm + 1):
        theta = torch.tensor(synth.draw_prior(synth.PRIOR_GW170817, W, 7), device="cuda")
        n0 = rb.kernel_launch_count()
        L, G = rb.loglike_grad(event, theta, mode=mode + "_shared")
        assert rb.kernel_launch_count() - n0 == 2
        l = rb.loglike(event, theta, mode=mode + "_shared")
        ref_L, ref_G = rb.loglike_grad(event, theta, mode=mode)
        assert torch.equal(L, ref_L) and torch.equal(G, ref_G) and torch.equal(l, rb.loglike(event, theta, mode=mode))
    a, b = (torch.tensor(synth.posterior_box(ev["theta_inj"], 9, seed=3), device="cuda", requires_grad=True) for _ in range(2))
    rb.rb_loglike(a, event, mode + "_shared").sum().backward()
    rb.rb_loglike(b, event, mode).sum().backward()
    assert torch.equal(a.grad, b.grad)
    event.free()


def test_mala_and_refusals():
    import torch
    import paper_2404_11397_gb300 as rb
    ev = small_event()
    event = rb.Event.from_synth(ev, n_bins=70)
    c = np.array(ev["theta_inj"], dtype=np.float64)
    c[9], c[12] = np.cos(c[9]), np.sin(c[12])
    half = np.array([0.01, 0.05, 0.02, 0.02, 250.0, 250.0, 20.0, 0.05, 0.5, 0.05, 0.5, 0.5, 0.2])
    lo, hi = c - half, c + half
    rng = np.random.Generator(np.random.Philox(5))
    z0 = torch.tensor(lo + (hi - lo) * rng.uniform(0.3, 0.7, (77, 13)), device="cuda")
    xi, u = (torch.tensor(x, device="cuda") for x in (rng.standard_normal((77, 13)), 1.0 - rng.random(77)))
    out = []
    for mode in ("mixed", "mixed_shared"):
        z = z0.clone()
        logp, gz = rb.mala_init(event, z, lo, hi, mode=mode)
        acc = rb.mala_step(event, z, logp, gz, 4e-4 * half, lo, hi, xi, u, mode=mode)
        out.append((z, logp, gz, acc))
    for x, y in zip(*out):
        assert torch.equal(x, y)
    theta = torch.tensor(synth.posterior_box(ev["theta_inj"], 4, seed=3), device="cuda")
    for call in (lambda: event.rebuild(mode="mixed_shared"), lambda: rb.rebuild_loglike_grad(event, theta, mode="mixed_shared"),
                 lambda: rb.loglike_full(event, theta, mode="mixed_shared"),
                 lambda: rb.loglike_grad_host(event, theta.cpu().numpy(), np.empty(4), mode="mixed_shared"),
                 lambda: rb.Server(mode="mixed_shared")):
        with pytest.raises(rb.RBError):
            call()
    event.free()
