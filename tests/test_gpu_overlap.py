"""Results written into the walkers' own memory, at the same address or shifted against
it, and MALA's answers into its uniform draws: as with separate buffers, bit for bit,
also where another kernel holds most SMs back, so that some blocks start late."""
import numpy as np
import pytest

import synth
from tests._events import small_event

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def setting():
    import torch
    import paper_2404_11397_gb300 as rb
    ev = small_event(T=64.0)
    event = rb.Event.from_synth(ev, n_bins=700)  # tables of a size that one block fills an SM
    W = 32 * torch.cuda.get_device_properties(0).multi_processor_count
    theta = torch.tensor(synth.posterior_box(ev["theta_inj"], W, seed=21), device="cuda")
    yield ev, event, theta
    event.free()


def _beside_another(call, event, theta):
    """call() on the current stream while a full-grid batch runs on another."""
    import torch
    import paper_2404_11397_gb300 as rb
    other = torch.cuda.Stream()
    torch.cuda.synchronize()
    rb.loglike_full(event, theta[:24], stream=other)
    call()
    torch.cuda.synchronize()


# offsets in doubles of the results from theta's first, as shares of theta's length
@pytest.mark.parametrize("at", [0.0, 0.5, 12.0 / 13.0])
@pytest.mark.parametrize("grad", [False, True])
def test_results_into_theta(setting, at, grad):
    import torch
    import paper_2404_11397_gb300 as rb
    from paper_2404_11397_gb300._lib import check
    _, event, theta = setting
    W = theta.shape[0]
    ref = rb.loglike_grad(event, theta) if grad else (rb.loglike(event, theta),)
    buf = torch.empty(theta.numel() * 3, dtype=torch.float64, device="cuda")
    t = buf[:theta.numel()].view(W, 13)
    o = int(at * theta.numel())
    if grad:  # log L apart, the gradient from theta's o-th double on
        L, G = torch.empty(W, dtype=torch.float64, device="cuda"), buf[o:o + 13 * W].view(W, 13)
    else:
        L, G = buf[o:o + W], None
    s = torch.cuda.current_stream().cuda_stream
    rb.loglike_full(event, theta[:24])
    t.copy_(theta)

    def call():
        if grad:
            check(rb.load().rb_loglike_grad_batch(event.handle, t.data_ptr(), W, L.data_ptr(), G.data_ptr(), 0, s), "call")
        else:
            check(rb.load().rb_loglike_batch(event.handle, t.data_ptr(), W, L.data_ptr(), 0, s), "call")

    _beside_another(call, event, theta)
    assert torch.equal(L, ref[0])
    if grad:
        assert torch.equal(G, ref[1])


def test_mala_answers_into_the_draws(setting):
    import torch
    import paper_2404_11397_gb300 as rb
    from paper_2404_11397_gb300._lib import check
    ev, event, theta = setting
    W = theta.shape[0]
    c = np.array(ev["theta_inj"], dtype=np.float64)
    c[9], c[12] = np.cos(c[9]), np.sin(c[12])
    half = np.array([0.01, 0.05, 0.02, 0.02, 250.0, 250.0, 20.0, 0.05, 0.5, 0.05, 0.5, 0.5, 0.2])
    lo, hi = c - half, c + half
    rng = np.random.Generator(np.random.Philox(5))
    z0 = torch.tensor(lo + (hi - lo) * rng.uniform(0.3, 0.7, (W, 13)), device="cuda")
    xi, u0 = (torch.tensor(x, device="cuda") for x in (rng.standard_normal((W, 13)), 1.0 - rng.random(W)))
    logp0, gz0 = rb.mala_init(event, z0, lo, hi)
    eps = 4e-4 * half
    z, logp, gz = z0.clone(), logp0.clone(), gz0.clone()
    ref = rb.mala_step(event, z, logp, gz, eps, lo, hi, xi, u0)
    z2, logp2, gz2, u = z0.clone(), logp0.clone(), gz0.clone(), u0.clone()
    acc = u.view(torch.int32)[W:]  # the int32 answers over the draws' second half
    s = torch.cuda.current_stream().cuda_stream
    _beside_another(lambda: check(rb.load().rb_mala_step(
        event.handle, z2.data_ptr(), logp2.data_ptr(), gz2.data_ptr(), W, eps.ctypes.data, lo.ctypes.data, hi.ctypes.data,
        xi.data_ptr(), u.data_ptr(), acc.data_ptr(), 0, s), "call"), event, theta)
    assert 0 < int(ref.sum()) < W
    assert torch.equal(acc, ref) and torch.equal(z2, z) and torch.equal(logp2, logp) and torch.equal(gz2, gz)
