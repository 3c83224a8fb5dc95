"""rb_kernel_launch_count while one thread captures host-buffer calls and others
launch batches: every call here is one kernel (a small mixed batch takes set-up and
likelihood in one launch), captures launch nothing, so the count is the number of calls."""
import threading

import pytest

import synth
from tests._events import small_event

pytestmark = pytest.mark.gpu


def test_captures_do_not_count_other_threads_launches():
    import torch
    import paper_2404_11397_gb300 as rb
    ev = small_event(sites=("H1",))
    events = [rb.Event.from_synth(ev, n_bins=70) for _ in range(2)]
    theta = synth.posterior_box(ev["theta_inj"], 64, seed=5)
    dev = torch.tensor(theta, device="cuda")
    host = torch.empty(theta.shape, dtype=torch.float64, pin_memory=True)
    host.copy_(torch.from_numpy(theta))
    logl = [torch.empty(64, dtype=torch.float64, pin_memory=True) for _ in range(2)]
    rb.loglike(events[1], dev)
    rb.loglike_grad_host(events[0], host, logl[0])
    torch.cuda.synchronize()
    start, calls, stop = rb.kernel_launch_count(), [0] * 4, threading.Event()

    def batches(k):  # the C call alone, so that its launches fall into the other thread's captures
        out, stream = torch.empty(64, dtype=torch.float64, device="cuda"), torch.cuda.Stream()
        call, args = rb.load().rb_loglike_batch, (events[1].handle, dev.data_ptr(), 64, out.data_ptr(), 0, stream.cuda_stream)
        while not stop.is_set():
            for _ in range(50):
                call(*args)
            calls[k] += 50
        stream.synchronize()

    threads = [threading.Thread(target=batches, args=(k,)) for k in range(len(calls))]
    for t in threads:
        t.start()
    try:
        n = 1000
        for i in range(n):  # other outputs than the call before: each is captured anew and launched
            rb.loglike_grad_host(events[0], host, logl[(i + 1) % 2])
    finally:
        stop.set()
        for t in threads:
            t.join()
    assert rb.kernel_launch_count() - start == n + sum(calls)
    for e in events:
        e.free()


def test_replays_of_one_event_from_two_threads():
    """Two threads replay one event's captured call, one with a batch of one kernel, the
    other with a batch of two: each replay counts its own."""
    import torch
    import paper_2404_11397_gb300 as rb
    ev = small_event(sites=("H1",))
    event = rb.Event.from_synth(ev, n_bins=70)
    sizes, each, per_call = (64, 40_000), 300, []
    for W in sizes:
        n0 = rb.kernel_launch_count()
        rb.loglike(event, torch.tensor(synth.posterior_box(ev["theta_inj"], W, seed=5), device="cuda"))
        per_call.append(rb.kernel_launch_count() - n0)
    assert per_call == [1, 2]
    start = rb.kernel_launch_count()

    def replays(W):
        host = torch.empty(W, 13, dtype=torch.float64, pin_memory=True)
        host.copy_(torch.from_numpy(synth.posterior_box(ev["theta_inj"], W, seed=5)))
        logl = torch.empty(W, dtype=torch.float64, pin_memory=True)
        for _ in range(each):
            rb.loglike_grad_host(event, host, logl)

    threads = [threading.Thread(target=replays, args=(W,)) for W in sizes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert rb.kernel_launch_count() - start == sum(per_call) * each
    event.free()
