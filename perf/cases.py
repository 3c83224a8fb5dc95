"""Performance cases: the work that users of this library have it do, through its public entry points.

A case is a dict of plain values: which call, the event (detectors, duration, band, bins), the walkers and the
evaluation mode.  ``prepare`` makes what a sampler has in hand before the call (a resident event, walkers, for the
host calls pinned buffers, for serving a running server), ``run`` makes one call and returns everything it computes,
``work`` counts what the call cannot do without, and ``exact`` gives the same results from plain FP64 torch and
numpy, written from the method's formulas and not from the library's code.

Sizes: the library's four reference workloads (1 detector, T = 64 s, 20-1024 Hz, 100 bins; 3 detectors, T = 128 s,
20-2048 Hz, 500 bins, 4096 walkers; the same with T = 256 s, 1000 bins, 16384 walkers; serving mixes of both), and
ragged sizes between them.
"""
import math

import numpy as np
import torch

import paper_2404_11397_gb300 as rb

# ---- sites, prior boxes, injection ------------------------------------------------------------------------------
# latitude, longitude [deg], elevation [m], x- and y-arm azimuths [deg clockwise from North]
SITES = [(46.455, -119.408, 142.554, 126.0, 216.0), (30.563, -90.774, -6.574, 197.7, 287.7),
         (43.631, 10.505, 51.884, 70.6, 160.6)]
GMST = 1.0
NPAR = 13
# (Mc, q, chi1, chi2, Lambda1, Lambda2, dL, tc, phic, iota, psi, ra, dec)
SOURCES = {
    "light": [1.17419, 0.92857, 0.02, 0.02, 300.0, 400.0, 40.0, 0.0, 1.0, 0.4, 0.6, 3.45, -0.41],
    "heavy": [1.44, 0.8, 0.02, 0.02, 800.0, 900.0, 40.0, 0.0, 1.0, 0.4, 0.6, 3.45, -0.41],
}
PRIORS = {  # lo, hi; iota and dec are drawn through cos(iota) and sin(dec)
    "light": ([1.18, 0.125, -0.05, -0.05, 0.0, 0.0, 1.0, -0.1, 0.0, -1.0, 0.0, 0.0, -1.0],
              [1.21, 1.0, 0.05, 0.05, 5000.0, 5000.0, 75.0, 0.1, 2 * math.pi, 1.0, math.pi, 2 * math.pi, 1.0]),
    "heavy": ([1.42, 0.125, -0.05, -0.05, 0.0, 0.0, 1.0, -0.1, 0.0, -1.0, 0.0, 0.0, -1.0],
              [1.46, 1.0, 0.05, 0.05, 3000.0, 3000.0, 75.0, 0.1, 2 * math.pi, 1.0, math.pi, 2 * math.pi, 1.0]),
}
WIDTH = np.array([0.03, 0.875, 0.1, 0.1, 5000.0, 5000.0, 74.0, 0.2, 2 * math.pi, math.pi, math.pi, 2 * math.pi, math.pi])


def _case(name, call, det, T, f_high, bins, walkers, box="prior", source="light", mode="mixed"):
    c = {"call": call, "det": det, "T": T, "f_low": 20.0, "f_high": f_high, "bins": bins, "walkers": walkers,
         "box": box, "source": source, "mode": mode}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: log L at a few tens of points (an optimiser's population on a short event)
        _case("logl_few", "loglike", 1, 64.0, 1024.0, 100, 48, box="box"),
        # one detector, 4096 walkers through torch autograd: forward and backward
        _case("autograd_1det", "autograd", 1, 64.0, 1024.0, 100, 4096, box="box"),
        # two detectors, ragged walker and bin counts: a run's odd-sized population near the posterior
        _case("grad_2det_ragged", "grad", 2, 96.0, 1792.0, 237, 777, box="posterior"),
        # the long event's sampler batch, the largest of the binned calls
        _case("grad_heavy", "grad", 3, 256.0, 2048.0, 1000, 16384, source="heavy"),
        # the whole step on resident data: summary rebuild, then log L and gradient of 4096 walkers
        _case("step", "step", 3, 128.0, 2048.0, 500, 4096),
        # the same step end to end: strain, PSD and walkers in from pinned host memory, results out to it
        _case("step_host", "step_host", 3, 128.0, 2048.0, 500, 4096),
        # a sampler on the host with the event resident: walkers in, log L and gradient out
        _case("batch_host", "batch_host", 3, 128.0, 2048.0, 500, 4096),
        # one local sampler step of 1000 chains near the posterior, the chains' last positions kept
        _case("mala", "mala", 3, 128.0, 2048.0, 200, 1000, box="posterior"),
        # the un-binned likelihood on the full grid: the search for the reference point
        _case("full_grid", "full", 3, 128.0, 2048.0, 500, 512),
        # a new reference point after that search: the FP64 summary data of the long event, read back
        _case("rebuild_fp64", "rebuild", 3, 256.0, 2048.0, 1000, 0, source="heavy", mode="fp64"),
        # the plain FP64 path with the gradient: the check of a run's mixed results
        _case("grad_fp64", "grad", 3, 128.0, 2048.0, 200, 1000, mode="fp64"),
        # serving: requests of many sizes for several resident events, in flight together
        _case("serve", "serve", 3, 128.0, 2048.0, 500, 2048),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["loglike", "autograd", "grad", "grad", "step", "step_host", "batch_host", "mala", "full", "rebuild",
                       "grad_fp64", "serve"])
    det = rng.choice([1, 2, 3])
    T = rng.choice([64.0, 96.0, 128.0, 256.0])
    f_high = rng.choice([1024.0, 1500.0, 1792.0, 2048.0])
    source = rng.choice(["light", "light", "heavy"])
    box = rng.choice(["prior", "prior", "posterior", "box"])
    bins = _log(rng, 50, 1000)
    if call == "loglike":
        return _case("", "loglike", det, T, f_high, bins, _log(rng, 1, 4096), box, source)
    if call == "autograd":
        return _case("", "autograd", det, T, f_high, bins, _log(rng, 64, 4096), box, source)
    if call == "grad":
        return _case("", "grad", det, T, f_high, bins, _log(rng, 16, 16384), box, source)
    if call in ("step", "step_host", "batch_host"):
        return _case("", call, det, T if call == "batch_host" else rng.choice([64.0, 96.0, 128.0]), f_high, bins,
                     _log(rng, 256, 4096), box, source)
    if call == "mala":
        return _case("", "mala", det, T, f_high, _log(rng, 50, 500), _log(rng, 100, 1000), "posterior", source)
    if call == "full":
        T = rng.choice([64.0, 96.0, 128.0])
        return _case("", "full", det, T, f_high, _log(rng, 50, 500), _log(rng, 16, 512), box, source)
    if call == "rebuild":
        return _case("", "rebuild", det, T, f_high, bins, 0, "prior", source, "fp64")
    if call == "grad_fp64":
        return _case("", "grad", det, T, f_high, _log(rng, 50, 200), _log(rng, 32, 1000), box, source, "fp64")
    return _case("", "serve", rng.choice([2, 3]), rng.choice([64.0, 128.0]), f_high, _log(rng, 100, 500),
                 _log(rng, 256, 2048), box, source)


# ---- inputs -----------------------------------------------------------------------------------------------------
def _grid(case):
    k0 = int(math.ceil(case["f_low"] * case["T"] - 1e-9))
    k1 = int(math.floor(case["f_high"] * case["T"] + 1e-9))
    return k0, k1 - k0 + 1


def _geometry(det):
    g = np.array(SITES[:det], dtype=np.float64)
    g[:, [0, 1, 3, 4]] = np.deg2rad(g[:, [0, 1, 3, 4]])
    return g


def _psd(f):
    """Analytic fit of the advanced-LIGO design curve (zero-detuned, high power)."""
    x = f / 245.4
    return 1e-49 * (x ** -4.14 - 5.0 * x ** -2 + 111.0 * (1.0 - x ** 2 + 0.5 * x ** 4) / (1.0 + 0.5 * x ** 2))


def _antenna(th, geom):
    """Complex prefactor [W, D] and delay t_c + dt [W, D] of walkers th [W, 13]."""
    lat, lon, elev, xa, ya = (torch.tensor(geom[:, i], device=th.device) for i in range(5))
    north = torch.stack([-torch.sin(lat) * torch.cos(lon), -torch.sin(lat) * torch.sin(lon), torch.cos(lat)], 1)
    east = torch.stack([-torch.sin(lon), torch.cos(lon), torch.zeros_like(lon)], 1)
    x = torch.cos(xa)[:, None] * north + torch.sin(xa)[:, None] * east
    y = torch.cos(ya)[:, None] * north + torch.sin(ya)[:, None] * east
    a, e2 = 6378137.0, 6.69437999014e-3
    R = a / torch.sqrt(1.0 - e2 * torch.sin(lat) ** 2)
    r = torch.stack([(R + elev) * torch.cos(lat) * torch.cos(lon), (R + elev) * torch.cos(lat) * torch.sin(lon),
                     (R * (1.0 - e2) + elev) * torch.sin(lat)], 1)
    iota, psi, ra, dec = (th[:, j] for j in (9, 10, 11, 12))
    g = GMST - ra
    sg, cg, sd, cd, sp, cp, ci = g.sin(), g.cos(), dec.sin(), dec.cos(), psi.sin(), psi.cos(), iota.cos()
    X = torch.stack([-cp * sg - sp * cg * sd, -cp * cg + sp * sg * sd, sp * cd], 1)
    Y = torch.stack([sp * sg - cp * cg * sd, sp * cg + cp * sg * sd, cp * cd], 1)
    xX, xY, yX, yY = X @ x.T, Y @ x.T, X @ y.T, Y @ y.T
    fp = 0.5 * (xX ** 2 - yX ** 2 - xY ** 2 + yY ** 2)
    fc = xX * xY - yX * yY
    n = torch.stack([cd * cg, -cd * sg, sd], 1)
    tau = th[:, 7:8] - (n @ r.T) / 299792458.0
    return torch.complex(fp * (0.5 * (1.0 + ci ** 2))[:, None], -fc * ci[:, None]), tau


def _phase_terms(th):
    """Coefficients [W, 10] of f^(-5/3, -1, -2/3, -1/3), ln f, f^1/3, f^1/3 ln f, f^(2/3, 5/3, 7/3), and the constant [W]."""
    Mc, q, c1, c2, L1, L2 = (th[:, j] for j in range(6))
    eta = q / (1.0 + q) ** 2
    X1, X2 = 1.0 / (1.0 + q), q / (1.0 + q)
    beta = (c1 * (113.0 * X1 ** 2 + 75.0 * eta) + c2 * (113.0 * X2 ** 2 + 75.0 * eta)) / 12.0
    sigma = eta * (474.0 / 48.0) * c1 * c2 + (486.0 / 96.0) * (X1 ** 2 * c1 ** 2 + X2 ** 2 * c2 ** 2)
    p2 = 3715.0 / 756.0 + 55.0 / 9.0 * eta
    p3 = -16.0 * math.pi + 4.0 * beta
    p4 = 15293365.0 / 508032.0 + 27145.0 / 504.0 * eta + 3085.0 / 72.0 * eta ** 2 - 10.0 * sigma
    p5 = math.pi * (38645.0 / 756.0 - 65.0 / 9.0 * eta)
    p6 = (11583231236531.0 / 4694215680.0 - 640.0 / 3.0 * math.pi ** 2 - 6848.0 / 21.0 * 0.577215664901532860606512
          + eta * (-15737765635.0 / 3048192.0 + 2255.0 / 12.0 * math.pi ** 2) + 76055.0 / 1728.0 * eta ** 2
          - 127825.0 / 1296.0 * eta ** 3)
    p7 = math.pi * (77096675.0 / 254016.0 + 378515.0 / 1512.0 * eta - 74045.0 / 756.0 * eta ** 2)
    p10 = (-288.0 + 264.0 * X1) * X1 ** 4 * L1 + (-288.0 + 264.0 * X2) * X2 ** 4 * L2

    def t12(X, L):
        return X ** 4 * L * (-15895.0 / 28.0 + 4595.0 / 28.0 * X + 5715.0 / 14.0 * X ** 2 - 325.0 / 7.0 * X ** 3)

    p12 = t12(X1, L1) + t12(X2, L2)
    lnMc = torch.log(math.pi * 4.925490947641266978e-6 * Mc)
    u = lnMc - 0.6 * torch.log(eta)  # ln(pi M)
    N0, a = 3.0 / 128.0 * torch.exp(-5.0 / 3.0 * lnMc), torch.exp(u / 3.0)
    c = torch.stack([N0, N0 * a ** 2 * p2, N0 * a ** 3 * p3, N0 * a ** 4 * p4, N0 * a ** 5 * p5,
                     N0 * a ** 6 * (p6 - 6848.0 / 21.0 * (math.log(4.0) + u / 3.0)), N0 * a ** 6 * (-6848.0 / 63.0),
                     N0 * a ** 7 * p7, N0 * a ** 10 * p10, N0 * a ** 12 * p12], 1)
    return c, -th[:, 8] - 0.25 * math.pi + N0 * a ** 5 * p5 * (1.0 + 1.5 * math.log(6.0) + u)


def _powers(f):
    lf, cf = torch.log(f), f ** (1.0 / 3.0)
    return torch.stack([1.0 / (f * cf ** 2), 1.0 / f, cf ** -2, 1.0 / cf, lf, cf, cf * lf, cf ** 2, f * cf ** 2, f ** 2 * cf])


def _amplitude(th):
    return math.sqrt(5.0 / 24.0) * math.pi ** (-2.0 / 3.0) * (4.925490947641266978e-6 * th[:, 0]) ** (5.0 / 6.0) / (
        th[:, 6] * (3.085677581491367e22 / 299792458.0))


def _strain(th, geom, f):
    """h [W, D, N] of walkers th on frequencies f, FP64."""
    c, p0 = _phase_terms(th)
    P, tau = _antenna(th, geom)
    x = (c @ _powers(f) + p0[:, None])[:, None, :] + 2.0 * math.pi * tau[:, :, None] * f
    return torch.polar(_amplitude(th)[:, None, None] * f ** (-7.0 / 6.0) * torch.ones_like(x), -x) * P[:, :, None]


def _source(case):
    return np.array(SOURCES[case["source"]], dtype=np.float64)


def _walkers(case, seed, W=None):
    rng = np.random.Generator(np.random.Philox(seed))
    W = case["walkers"] if W is None else W
    u = rng.random((W, NPAR))
    c = _source(case)
    if case["box"] == "prior":
        lo, hi = (np.array(v) for v in PRIORS[case["source"]])
        th = lo + (hi - lo) * u
        th[:, 9], th[:, 12] = np.arccos(th[:, 9]), np.arcsin(th[:, 12])
        return th
    if case["box"] == "box":  # within 1 % of the source
        half = np.maximum(np.abs(c) * 0.01, 0.01 * WIDTH * (c == 0.0))
    else:  # the posterior's scale
        half = np.abs(c) * 1e-3
        half[0] = c[0] * 1e-5
        half = np.maximum(half, 1e-3 * WIDTH * (c == 0.0))
    th = c + (2.0 * u - 1.0) * half
    th[:, 1] = np.minimum(th[:, 1], 1.0)
    return th


def _data(case, seed, device):
    """Strain [D, N] complex and PSD [D, N]: the source's signal in seeded Gaussian noise."""
    k0, N = _grid(case)
    f = torch.arange(k0, k0 + N, dtype=torch.float64, device=device) / case["T"]
    geom = _geometry(case["det"])
    g = torch.Generator(device=device).manual_seed(int(seed))
    psd = torch.stack([_psd(f) * s for s in (1.0, 1.3, 2.5)[:case["det"]]])
    z = torch.randn(2, case["det"], N, dtype=torch.float64, device=device, generator=g)
    h = _strain(torch.tensor(_source(case), device=device)[None], geom, f)[0]
    return f, geom, psd, torch.complex(z[0], z[1]) * torch.sqrt(psd * (case["T"] / 4.0)) + h


def _event(case, seed):
    f, geom, psd, data = _data(case, seed, "cuda")
    ev = rb.Event(geom, GMST, case["T"], case["f_low"], case["f_high"], list(data), list(psd), case["bins"], _source(case))
    return ev, data, psd


def _new_reference(case, seed):
    return _walkers(dict(case, box="posterior"), seed + 7, 1)[0]


def _pinned(t):
    p = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    p.copy_(t)
    return p


# serving: per event (detectors, T as a share of the case's, bins as a share), then the requests (event, walkers as a share)
SERVED = [(0, 1.0, 1.0), (1, 1.0, 0.4), (0, 0.5, 0.7), (1, 0.5, 0.2)]
REQUESTS = [(0, 1.0), (1, 0.5), (2, 0.125), (3, 0.6), (0, 0.2), (1, 1.0), (2, 0.8), (3, 0.3), (0, 0.45), (2, 0.35)]


def _serve_parts(case, seed):
    evs = [dict(case, det=max(2, case["det"] - d), T=max(64.0, case["T"] * t), bins=max(20, int(case["bins"] * b)))
           for d, t, b in SERVED]
    reqs = [(e, _walkers(case, seed + 101 + i, max(16, int(case["walkers"] * w)))) for i, (e, w) in enumerate(REQUESTS)]
    return evs, reqs


def prepare(case, seed):
    call = case["call"]
    if call == "serve":
        evs, reqs = _serve_parts(case, seed)
        return {"case": case, "events": [_event(c, seed + i)[0] for i, c in enumerate(evs)], "reqs": reqs,
                "server": rb.Server(max_slots=4, max_walkers=8192, mode=case["mode"])}
    ev, data, psd = _event(case, seed)
    s = {"case": case, "event": ev}
    W = case["walkers"]
    if call == "rebuild":
        s["ref"] = _new_reference(case, seed)
        return s
    th = _walkers(case, seed + 1)
    if call in ("step_host", "batch_host"):
        s["theta"], s["logl"] = _pinned(torch.from_numpy(th)), torch.empty(W, dtype=torch.float64, pin_memory=True)
        s["grad"] = torch.empty(W, NPAR, dtype=torch.float64, pin_memory=True)
        if call == "step_host":
            s["data"] = [_pinned(torch.view_as_real(d).cpu()) for d in data]
            s["psd"] = [_pinned(p.cpu()) for p in psd]
        return s
    if call == "mala":
        lo, hi, eps, z, xi, u = _mala_inputs(case, seed)
        s["lo"], s["hi"], s["eps"] = lo, hi, eps
        s["z"], s["xi"], s["u"] = (torch.from_numpy(a).cuda() for a in (z, xi, u))
        s["logp"], s["gz"] = rb.mala_init(ev, s["z"], lo, hi, mode=case["mode"])
        return s
    s["theta"] = torch.from_numpy(th).cuda()
    if call == "autograd":
        s["theta"].requires_grad_(True)
    return s


def _mala_inputs(case, seed):
    z = _walkers(case, seed + 1)
    z[:, 9], z[:, 12] = np.cos(z[:, 9]), np.sin(z[:, 12])
    c = _source(case)
    c[9], c[12] = math.cos(c[9]), math.sin(c[12])
    half = np.array([0.01, 0.05, 0.02, 0.02, 250.0, 250.0, 20.0, 0.05, 0.5, 0.05, 0.5, 0.5, 0.2])
    lo, hi = c - half, np.array(c + half)
    eps = 4e-4 * half
    eps[0] = 4e-7
    rng = np.random.Generator(np.random.Philox(seed + 3))
    return lo, hi, eps, z, rng.standard_normal(z.shape), 1.0 - rng.random(z.shape[0])


def run(state):
    case = state["case"]
    call, mode = case["call"], case["mode"]
    if call == "loglike":
        return rb.loglike(state["event"], state["theta"], mode=mode)
    if call == "grad":
        return rb.loglike_grad(state["event"], state["theta"], mode=mode)
    if call == "autograd":
        theta = state["theta"]
        theta.grad = None
        logl = rb.rb_loglike(theta, state["event"], mode)
        logl.sum().backward()
        return logl.detach(), theta.grad
    if call == "step":
        return rb.rebuild_loglike_grad(state["event"], state["theta"], mode=mode)
    if call == "step_host":
        rb.rebuild_loglike_grad_host(state["event"], state["data"], state["psd"], state["theta"], state["logl"],
                                     state["grad"], mode=mode)
        return state["logl"], state["grad"]
    if call == "batch_host":
        rb.loglike_grad_host(state["event"], state["theta"], state["logl"], state["grad"], mode=mode)
        return state["logl"], state["grad"]
    if call == "mala":
        z, logp, gz = state["z"].clone(), state["logp"].clone(), state["gz"].clone()
        acc = rb.mala_step(state["event"], z, logp, gz, state["eps"], state["lo"], state["hi"], state["xi"], state["u"],
                           mode=mode)
        return z, logp, gz, acc
    if call == "full":
        return rb.loglike_full(state["event"], state["theta"], mode=mode)
    if call == "rebuild":
        state["event"].rebuild(theta_ref=state["ref"], mode=mode)
        return state["event"].summary()
    srv = state["server"]
    tickets = [srv.submit(state["events"][e], th) for e, th in state["reqs"]]
    return [srv.poll(t)[1:] for t in tickets]


# ---- the work that cannot be left out ----------------------------------------------------------------------------
def _batch_work(D, B, W, grad):
    """One walker and edge: ten phase terms; per detector the delay, a sine and cosine (~30), the ratio and the bin's
    contraction (~28); with the gradient the cotangents (~26) and ten products back to the phase terms."""
    per = 20 + 60 * D + ((26 * D + 20) if grad else 0)
    return {"flops": float(W * (B + 1) * per), "bytes": 8.0 * (W * (NPAR + 1 + (NPAR if grad else 0)) + 11 * (B + 1) + 6 * D * B)}


def work(case):
    D, B, W, call = case["det"], case["bins"], case["walkers"], case["call"]
    _, N = _grid(case)
    if call == "serve":
        evs, reqs = _serve_parts(case, 0)
        parts = [_batch_work(evs[e]["det"], evs[e]["bins"], th.shape[0], True) for e, th in reqs]
        return {k: sum(p[k] for p in parts) for k in ("flops", "bytes")}
    # the summary: strain and PSD read; per point the phase (20), a sine and cosine, per detector the six sums (~30)
    summary = {"flops": float(N * (50 + 30 * D)), "bytes": 24.0 * N * D + 48.0 * D * B}
    if call == "rebuild":
        return summary
    if call == "full":  # per walker and point: the phase, a sine and cosine, per detector the delay and the product
        return {"flops": float(W * N * (50 + 12 * D)), "bytes": 24.0 * N * D + 8.0 * W * (NPAR + 1)}
    w = _batch_work(D, B, W, call != "loglike")
    if call in ("step", "step_host"):
        w = {k: w[k] + summary[k] for k in w}
    if call == "mala":
        w["bytes"] += 8.0 * W * (4 * NPAR + 4)
    return w


# ---- the same results in plain FP64 -------------------------------------------------------------------------------
def _edges(case):
    """Bin edges equally spaced in the post-Newtonian phase bound, on the grid."""
    k0, N = _grid(case)
    B = case["bins"]
    f = np.arange(k0, k0 + N, dtype=np.float64) / case["T"]
    P = 2.0 * math.pi * sum((1.0 if g > 0 else -1.0) * (f / (case["f_high"] if g > 0 else case["f_low"])) ** g
                            for g in (-5.0 / 3.0, -2.0 / 3.0, 1.0, 5.0 / 3.0, 7.0 / 3.0))
    tau = P[0] + (P[-1] - P[0]) * np.arange(B + 1) / B
    k = np.minimum(np.searchsorted(P, tau, side="right") - 1, N - 2)
    e = np.where((tau - P[k]) / (P[k + 1] - P[k]) < 0.5, k, k + 1)
    e[0], e[-1] = 0, N - 1
    i = np.arange(B + 1)
    return i + np.maximum.accumulate(np.clip(e, i, N - 1 - (B - i)) - i)


def _summary(case, seed, ref, device):
    """A0, A1 (complex), B0, B1 [D, B], the edges' frequencies and the bin widths."""
    f, geom, psd, data = _data(case, seed, device)
    edges = torch.from_numpy(_edges(case)).to(device)
    B = case["bins"]
    h0 = _strain(torch.tensor(ref, device=device)[None], geom, f)[0]
    b = torch.clamp(torch.searchsorted(edges, torch.arange(f.numel(), device=device), right=True) - 1, max=B - 1)
    fe = f[edges]
    fm = 0.5 * (fe[1:] + fe[:-1])
    df = f - fm[b]
    w = (4.0 / case["T"]) / psd
    x, hh = data * h0.conj() * w, h0.abs() ** 2 * w

    def total(v):
        return torch.zeros(v.shape[0], B, dtype=torch.float64, device=device).index_add_(1, b, v)

    out = {"B0": total(hh), "B1": total(hh * df)}
    for name, v in (("A0", x), ("A1", x * df)):
        out[name] = torch.complex(total(v.real.contiguous()), total(v.imag.contiguous()))
    return out, geom, fe, edges


def _binned(s, geom, fe, ref, th, grad, device):
    """log L [W] and its gradient [W, 13] of walkers th (numpy) from the summary data."""
    r13 = torch.tensor(ref, device=device)[None]
    g = _powers(fe)
    c0, p00 = _phase_terms(r13)
    P0, t0 = _antenna(r13, geom)
    df = fe[1:] - fe[:-1]
    logl, gr = [], []
    step = max(1, 6_000_000 // (fe.numel() * len(geom)))
    for i in range(0, len(th), step):
        t = torch.tensor(th[i:i + step], device=device).requires_grad_(grad)
        with torch.set_grad_enabled(grad):
            c, p0 = _phase_terms(t)
            P, tau = _antenna(t, geom)
            x = ((c - c0) @ g + (p0 - p00)[:, None])[:, None, :] + 2.0 * math.pi * (tau - t0)[:, :, None] * fe
            rho = (_amplitude(t) / _amplitude(r13))[:, None] * P / P0
            r = rho[:, :, None] * torch.complex(torch.cos(x), -torch.sin(x))
            r0, r1 = 0.5 * (r[..., 1:] + r[..., :-1]), (r[..., 1:] - r[..., :-1]) / df
            v = (s["A0"] * r0.conj() + s["A1"] * r1.conj()).real - 0.5 * (
                s["B0"] * (r0.real ** 2 + r0.imag ** 2) + 2.0 * s["B1"] * (r0 * r1.conj()).real)
            L = v.sum((1, 2))
        if grad:
            gr.append(torch.autograd.grad(L.sum(), t)[0])
        logl.append(L.detach())
    return torch.cat(logl), torch.cat(gr) if grad else None


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    call, ref = case["call"], _source(case)
    if call == "serve":
        evs, reqs = _serve_parts(case, seed)
        sums = [_summary(c, seed + i, ref, device) for i, c in enumerate(evs)]
        return [list(_binned(*sums[e][:3], ref, th, True, device)) for e, th in reqs]
    if call == "rebuild":
        s, _, _, edges = _summary(case, seed, _new_reference(case, seed), device)
        return dict(s, edges=edges)
    if call == "full":
        f, geom, psd, data = _data(case, seed, device)
        w, out = (4.0 / case["T"]) / psd, []
        th = torch.tensor(_walkers(case, seed + 1), device=device)
        step = max(1, 8_000_000 // data.numel())
        for i in range(0, len(th), step):
            h = _strain(th[i:i + step], geom, f)
            out.append(((data * h.conj()).real * w - 0.5 * (h.real ** 2 + h.imag ** 2) * w).sum((1, 2)))
        return torch.cat(out)
    s, geom, fe, _ = _summary(case, seed, ref, device)
    if call == "mala":
        return _exact_mala(case, seed, s, geom, fe, ref, device)
    logl, grad = _binned(s, geom, fe, ref, _walkers(case, seed + 1), call != "loglike", device)
    return logl if call == "loglike" else [logl, grad]


def _exact_mala(case, seed, s, geom, fe, ref, device):
    lo, hi, eps, z, xi, u = _mala_inputs(case, seed)

    def target(z):
        inside = np.all((z > lo) & (z < hi), axis=1)
        th = np.array(z)
        th[:, 9], th[:, 12] = np.arccos(th[:, 9]), np.arcsin(th[:, 12])
        logl, g = _binned(s, geom, fe, ref, th, True, device)
        g = g.cpu().numpy()
        g[:, 9] *= -1.0 / np.sqrt((1.0 - z[:, 9]) * (1.0 + z[:, 9]))
        g[:, 12] *= 1.0 / np.sqrt((1.0 - z[:, 12]) * (1.0 + z[:, 12]))
        return np.where(inside, logl.cpu().numpy(), -np.inf), np.where(inside[:, None], g, 0.0)

    logp, gz = target(z)
    zp = z + 0.5 * eps ** 2 * gz + eps * xi
    zc = np.where(np.all((zp > lo) & (zp < hi), axis=1)[:, None], zp, z)
    logpp, gzp = target(zc)
    inside = np.all((zp > lo) & (zp < hi), axis=1)
    la = np.where(inside, logpp - logp - 0.5 * np.sum((xi + 0.5 * eps * (gz + gzp)) ** 2 - xi ** 2, axis=1), -np.inf)
    acc = np.log(u) < la
    return [np.where(acc[:, None], zp, z), np.where(acc, logpp, logp), np.where(acc[:, None], gzp, gz), None]
