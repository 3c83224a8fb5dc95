"""A saved event loads to the bits of its FP64 summary, whichever way h0 was generated:
at every point (created at r, or moved to r by a mixed rebuild and then rebuilt in FP64) or
from Taylor chunks (rebuilt to r in FP64, k_min from 1024 on), also when the loaded event
is saved again, and where a file does not say (written before there was a choice) as
at creation.  The two ways agree within FP64 rounding: phases of ~1e4 rad carry 1e-12, 1e-10 of
a detector's largest entry taken."""
import numpy as np
import pytest

import synth
from tests._events import inject

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,f_high", [(64.0, 300.0), (8.0, 300.0)])
@pytest.mark.parametrize("sites", [("H1",), ("H1", "V1"), ("H1", "L1", "V1")])
def test_a_saved_event_loads_to_its_own_bits(sites, T, f_high, tmp_path):
    import torch
    import paper_2404_11397_gb300 as rb
    ev = inject(synth.make_event("C2", T=T, f_high=f_high, sites=sites))
    ref = synth.posterior_box(ev["theta_inj"], 1, seed=17)[0]
    th = torch.tensor(synth.posterior_box(ev["theta_inj"], 40, seed=18), device="cuda")

    def state(e):
        L, G = rb.loglike_grad(e, th, mode="fp64")
        return {**e.summary(), "base": e.info()["base_logl"], "L": L.cpu().numpy(), "G": G.cpu().numpy()}

    def equal(a, b):
        for k in a:
            np.testing.assert_array_equal(a[k], b[k], err_msg=k)

    created = rb.Event.from_synth(ev, n_bins=60, theta_ref=ref)
    rebuilt = rb.Event.from_synth(ev, n_bins=60)
    rebuilt.rebuild(theta_ref=ref, mode="fp64")
    mixed = rb.Event.from_synth(ev, n_bins=60)
    mixed.rebuild(theta_ref=ref, mode="mixed")
    if ev["kmin"] >= 1024:  # (below, that was an FP64 build already, whose h0 the next one would stream in another order)
        mixed.rebuild(mode="fp64")
    states = []
    for i, e in enumerate((created, rebuilt, mixed)):
        own = state(e)
        path = tmp_path / str(i)
        for _ in range(2):
            e.save(path)
            e.free()
            e = rb.Event.load(path)
            equal(own, state(e))
        e.free()
        states.append(own)
    # created and moved in two steps: the same edges and the same evaluation at every point
    edges = states[0]["edges"]
    for s in states[1:]:
        if np.array_equal(s["edges"], edges):
            for k in ("A0", "A1", "B0", "B1"):
                scale = np.max(np.abs(states[0][k]), axis=1, keepdims=True)
                assert np.max(np.abs(s[k] - states[0][k]) / scale) <= 1e-10, k
    # a file that does not say: the evaluation at every point
    raw = bytearray((tmp_path / "1").read_bytes())
    D, N = ev["psd"].shape
    at = len(raw) - 24 * D * N - 4  # the header's last field, in front of strain and PSD
    assert int.from_bytes(raw[at:at + 4], "little") == (1 if ev["kmin"] >= 1024 else 0)
    raw[at:at + 4] = bytes(4)
    (tmp_path / "old").write_bytes(raw)
    old = rb.Event.load(tmp_path / "old")
    equal(states[0], state(old))
    old.free()
