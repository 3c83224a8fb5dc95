"""Device strain and PSD read in place from addresses that are multiples of 8 bytes only
(slices of a larger buffer): every rebuild gives the bits it gives for copies on
16-byte boundaries."""
import numpy as np
import pytest

import synth
from tests._events import inject

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sites", [("H1",), ("H1", "L1"), ("H1", "L1", "V1")])
@pytest.mark.parametrize("T", [64.0, 8.0])
def test_unaligned_in_place_data(sites, T):
    import torch
    import paper_2404_11397_gb300 as rb
    ev = inject(synth.make_event("C2", T=T, f_high=300.0, sites=sites))
    D, N = ev["psd"].shape
    ref = synth.posterior_box(ev["theta_inj"], 1, seed=4)[0]
    data = np.stack([ev["data"].real, ev["data"].imag], -1) * 0.75

    def placed(shift):
        buf = torch.empty(3 * D * N + 1, dtype=torch.float64, device="cuda")
        d, p = buf[shift:shift + 2 * D * N].view(D, N, 2), buf[shift + 2 * D * N:shift + 3 * D * N].view(D, N)
        d.copy_(torch.from_numpy(data))
        p.copy_(torch.from_numpy(ev["psd"]))
        assert d.data_ptr() % 16 == 8 * shift
        return list(d), list(p)

    out = []
    for shift in (0, 1):
        event = rb.Event.from_synth(ev, n_bins=40)
        d, p = placed(shift)
        s = []
        for kw in (dict(theta_ref=ref, mode="fp64"), dict(mode="fp64"), dict(mode="mixed"),
                   dict(theta_ref=ev["theta_inj"], mode="mixed"), dict(mode="fp64")):
            event.rebuild(data=d, psd=p, **kw)
            s.append({**event.summary(), "base": event.info()["base_logl"]})
        event.free()
        out.append(s)
    for a, b in zip(*out):
        for k in a:
            np.testing.assert_array_equal(a[k], b[k], err_msg=k)
