"""FP64 log L and gradient of walkers whose phases are far beyond 2^49 turns (RB_FP64
has no phase limit).  theta_ref with a t_c of 1e16 s and more: the detectors' delays
are lost in t_c's rounding, and every product f t_c is beyond 2^53, so that every
phase difference is a whole number of turns and the results are theta_ref's own.
Tolerance: the ratio is 1 up to the rounding of the prefactors (a few 2^-53), so
log L differs by 1e-14 of its terms and the gradient by 1e-14 of the terms of its sums; 1e-11 taken.

A fiducial waveform with such a t_c keeps its modulus: by Cauchy-Schwarz no bin's |A0|
exceeds sqrt(<d|d> <h0|h0>) of the bin (1e-12 for the sums' rounding).  At the second
t_c, eight grid steps are just below a power of two of turns, where the sum with the
reduction's rounding constant loses the most."""
import numpy as np
import pytest

from tests._events import small_event

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sites", [("H1",), ("H1", "L1", "V1")])
@pytest.mark.parametrize("tc", [1e16, 3.0 ** 35, 1e20, 7.0 ** 40])
def test_whole_turns_leave_no_trace(sites, tc):
    import torch
    import paper_2404_11397_gb300 as rb
    ev = small_event(sites=sites)
    event = rb.Event.from_synth(ev, n_bins=70)
    theta = np.tile(ev["theta_inj"], (3, 1))
    theta[1, 7], theta[2, 7] = tc, -tc
    L, G = (x.cpu().numpy() for x in rb.loglike_grad(event, torch.tensor(theta, device="cuda"), mode="fp64"))
    s = event.summary()
    scale = np.sum(np.abs(s["A0"])) + np.sum(np.abs(s["B0"]))
    assert np.all(np.abs(L - event.info()["base_logl"]) <= 1e-11 * scale)
    # the same sums with the same tangents (they do not depend on t_c)
    tangent = np.maximum(np.abs(G[0]), 2 * np.pi * ev["f"][-1])
    assert np.all(np.abs(G[1:] - G[0]) <= 1e-11 * scale * tangent)
    event.free()


@pytest.mark.parametrize("tc", [1e16, 2.0 ** 61 - 64 * (2.0 ** 20 + 4), 1e20])
def test_far_reference_keeps_its_modulus(tc):
    import paper_2404_11397_gb300 as rb
    ev = small_event(T=64.0, f_high=200.0)
    event = rb.Event.from_synth(ev, n_bins=70)
    ref = np.array(ev["theta_inj"], dtype=np.float64)
    ref[7] = tc
    event.rebuild(theta_ref=ref, mode="fp64")
    s = event.summary()
    w = 4.0 / 64.0 * np.abs(ev["data"]) ** 2 / ev["psd"]
    dd = np.stack([np.add.reduceat(x, s["edges"][:-1]) for x in w])
    assert np.all(np.abs(s["A0"]) <= np.sqrt(dd * s["B0"]) * (1.0 + 1e-12))
    event.free()
