#!/usr/bin/env python3
"""Benchmark: relative-binning log-likelihood + gradient evaluations per second.

Workload (one step): the 3-detector event (H1/L1/V1-like sites, T = 128 s,
20-2048 Hz, 259,585 grid points, 500 bins, TaylorF2 + tides) with 4096 walkers
drawn from the GW170817 prior box.  A step runs the whole hot path: the
event's summary data are rebuilt from the strain and PSD resident in HBM
(fiducial waveform on the full grid, per-bin sums, tables; rb_event_rebuild),
then log L and its 13-parameter gradient are evaluated for the 4096 walkers
(rb_loglike_grad_batch).  Inputs are synthetic (seeded noise coloured by an
analytic aLIGO-like PSD plus an injected signal made by the library's strain
kernel).  L2 is flushed (a 256 MiB write) before every timed step.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl gb300|reference]

N > 1 runs one independent replica per GPU (launched by torch.distributed.run):
walkers are independent, so there is no data-path collective; rank 0 prints
one JSON line with the whole-job throughput over the slowest rank's time.
"""
from __future__ import annotations

import argparse
import json
import math
import os
import subprocess
import sys
import threading
import time
from pathlib import Path

import numpy as np

ROOT = Path(__file__).resolve().parent
sys.path.insert(0, str(ROOT))

METRIC = "RB logL+grad evals/sec (3 det, 4096 walkers) vs FP64 plain path; p50/p99 latency"
UNIT = "evals/s"
WORKLOAD = "3det_T128_f20-2048_500bins_4096walkers_TF2tidal_prior_GW170817"
N_SM = 152
FP32_LANES_PER_SM = 128
SM_MAX_MHZ = 2070.0


def parse():
    p = argparse.ArgumentParser()
    p.add_argument("--gpus", type=int, default=1)
    p.add_argument("--steps", type=int, default=200)
    p.add_argument("--warmup", type=int, default=10)
    p.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    p.add_argument("--mode", default="mixed", choices=["mixed", "mixed_f64phase", "fp64"])
    p.add_argument("--no-e2e", action="store_true")
    p.add_argument("--no-cpu", action="store_true")
    p.add_argument("--no-serving", action="store_true")
    p.add_argument("--no-mala", action="store_true")
    p.add_argument("--no-full", action="store_true")
    p.add_argument("--no-fp64", action="store_true")
    p.add_argument("--no-summary-build", action="store_true")
    p.add_argument("--no-configs", action="store_true", help="skip the C1 / C3 / C4 and FP64-phase legs")
    p.add_argument("--profile", action="store_true",
                   help="fixed short warm-up and no extra legs (for profiler launch lists)")
    return p.parse_args()


# ---------------------------------------------------------------------------
# Distributed helpers (replicas only)
# ---------------------------------------------------------------------------
class Dist:
    def __init__(self):
        self.world = int(os.environ.get("WORLD_SIZE", "1"))
        self.rank = int(os.environ.get("RANK", "0"))
        self.local = int(os.environ.get("LOCAL_RANK", "0"))
        self.pg = None

    def init(self, backend):
        if self.world > 1:
            import torch.distributed as dist
            dist.init_process_group(backend=backend)
            self.pg = dist

    def barrier(self):
        if self.pg:
            self.pg.barrier()

    def max(self, x: float, device) -> float:
        if not self.pg:
            return x
        import torch
        t = torch.tensor([x], dtype=torch.float64, device=device)
        self.pg.all_reduce(t, op=self.pg.ReduceOp.MAX)
        return float(t.item())

    def sum(self, x: float, device) -> float:
        if not self.pg:
            return x
        import torch
        t = torch.tensor([x], dtype=torch.float64, device=device)
        self.pg.all_reduce(t, op=self.pg.ReduceOp.SUM)
        return float(t.item())

    def close(self):
        if self.pg:
            self.pg.destroy_process_group()


def whole_job_rate(dist: Dist, total_s: float, units_per_rank: float, device=None):
    """Whole-job throughput of N independent replicas (weak scaling): every
    rank processes units_per_rank units; the job time is the slowest rank's
    timed total.  Returns (max_total_s, units of all ranks / max_total_s)."""
    max_total_s = dist.max(total_s, device)
    return max_total_s, units_per_rank * dist.world / max_total_s


# ---------------------------------------------------------------------------
# Clock sampling during the timed region
# ---------------------------------------------------------------------------
class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                                          "-lms", "100"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
            return
        self.t = threading.Thread(target=self._read, daemon=True)
        self.t.start()

    def _read(self):
        for ln in self.proc.stdout:
            self.lines.append(ln.strip())

    def stop(self) -> dict:
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"], "samples": 0}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.t.join(timeout=2)
        mhz, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [x.strip() for x in ln.split(",")]
            if len(parts) < 9 or parts[0] != str(self.gpu):
                continue
            try:
                mhz.append(float(parts[1]))
                mx.append(float(parts[2]))
            except ValueError:
                continue
            for n, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(n)
        return {"sm_mhz": float(np.median(mhz)) if mhz else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": sorted(reasons), "samples": len(mhz)}


# ---------------------------------------------------------------------------
# Algorithmic work of the relative-binning likelihood per walker (D detectors,
# B bins, E = B + 1 edges, K = 10 phase-basis functions as built), counted
# from the method, not from this implementation:
#   FP64-class: the basis dot product E * 2K, the delay term and range
#     reduction 8 D E, the per-walker set-up ~300; the gradient adds E K;
#   FP32-class: r0, r1 and the contraction 22 D B, the complex scaling of the
#     ratio 6 D E; the gradient triples it;
#   SFU: one sin/cos per (edge, detector).
# The mixed path runs all three classes on the FP32 pipe (FP64-class work as
# float-float), so the roofline adds them and divides by the FP32 peak.
# ---------------------------------------------------------------------------
N_BASIS = 10


def algorithmic_work(D: int, B: int, grad: bool) -> dict:
    E = B + 1
    fp64 = E * 2 * N_BASIS + 8 * D * E + 300 + (E * N_BASIS if grad else 0)
    fp32 = (22 * D * B + 6 * D * E) * (3 if grad else 1)
    sfu = D * E
    return {"fp64": fp64, "fp32": fp32, "sfu_sincos": sfu, "total": fp64 + fp32 + sfu}


# This implementation's own FP32 flop count of the same kernel (the float-pair
# emulation of the FP64-class work included), reported beside the algorithmic one.
def impl_flops_per_walker(D: int, B: int, grad: bool) -> int:
    # FP32 flops the mixed kernel spends per walker (FMA = 2): per edge the
    # float-pair phase sum (11 per basis term: high part rounded to the
    # walker's quantum, exact high sum, low sum); per edge and detector the
    # delay term and reduction to [-1/2, 1/2] (15), sin/cos (30), the ratio and
    # the bin's term (26); with the gradient the edge cotangents and adjoint
    # sums (22 per edge and detector, 20 per edge)
    E = B + 1
    f = E * 110 + D * E * 71
    if grad:
        f += D * E * 22 + E * 20
    return f


# DRAM bytes (dram__bytes_read.sum + dram__bytes_write.sum) of one launch of
# the main kernel on this workload, from an ncu capture of this kernel version
# (None once the kernel changes and until it is captured again).
MAIN_KERNEL_TRAFFIC_BYTES = 2391552


# Algorithmic FP32 flops of the full-grid sum per (walker, grid point) with 3
# detectors: the phase polynomial (30), one sin/cos (20), and per detector the
# delay rotation, the product with the data and the accumulation (14 each).
FULL_FLOPS_PER_WALKER_POINT = 92


def fp32_peak_tflops() -> float:
    """Derived from the unit counts and the maximum SM clock."""
    return N_SM * FP32_LANES_PER_SM * 2 * SM_MAX_MHZ * 1e6 / 1e12


# FFMA issue rate measured on this GPU by a microbenchmark (lane operations per
# clock per SM): 117.6 of the nominal 128.
FFMA_LANE_OPS_PER_CLK_SM = 117.6
# FP64 pipe: about 1.58 lane operations per clock per SM measured the same way.
FP64_LANE_OPS_PER_CLK_SM = 1.58


def ffma_measured_tflops() -> float:
    return N_SM * FFMA_LANE_OPS_PER_CLK_SM * 2 * SM_MAX_MHZ * 1e6 / 1e12


def fp64_measured_tflops() -> float:
    return N_SM * FP64_LANE_OPS_PER_CLK_SM * 2 * SM_MAX_MHZ * 1e6 / 1e12


def roofline_main(W: int, D: int, B: int, grad: bool, main_s: float) -> dict:
    """Main kernel against the FP32-pipe roofline with the method's algorithmic work."""
    work = algorithmic_work(D, B, grad)
    achieved = W * work["total"] / main_s / 1e12
    peak = fp32_peak_tflops()
    impl = impl_flops_per_walker(D, B, grad)
    return {"bound": "alu", "kernel": "k_rb_mixed (FP32 pipe)", "achieved": achieved, "peak": peak,
            "unit": "TFLOP/s", "frac": achieved / peak, "traffic": MAIN_KERNEL_TRAFFIC_BYTES if grad else None,
            "peak_source": "derived: 152 SMs x 128 FP32 lanes x 2 flop x 2070 MHz",
            "work_per_walker": work, "work_source": "algorithmic: FP64-class + FP32-class flops + sin/cos per walker",
            "peak_measured_ffma": ffma_measured_tflops(), "frac_of_measured_ffma": achieved / ffma_measured_tflops(),
            "fp64_class_tflops": W * work["fp64"] / main_s / 1e12,
            "fp64_class_frac_of_fp64_pipe": W * work["fp64"] / main_s / 1e12 / fp64_measured_tflops(),
            "impl_flops_per_walker": impl, "impl_tflops": W * impl / main_s / 1e12,
            "impl_frac": W * impl / main_s / 1e12 / peak}


# ---------------------------------------------------------------------------
def make_inputs(rb, torch, device, cfg="C2"):
    import synth
    ev = synth.make_event(cfg)
    D, N = ev["geom"].shape[0], ev["N"]
    # inject the signal with the library's own strain kernel (on the device)
    noise = torch.tensor(np.stack([ev["noise"].real, ev["noise"].imag], -1), device=device)
    data = torch.empty(D, N, 2, dtype=torch.float64, device=device)
    for d in range(D):
        h = rb.strain(ev["geom"][d], ev["gmst"], ev["theta_inj"], ev["T"], ev["kmin"], N, device=device)
        data[d] = noise[d] + torch.view_as_real(h)
    psd = torch.tensor(ev["psd"], device=device)
    torch.cuda.synchronize()
    return ev, data, psd


def run_gb300(args, dist: Dist):
    import torch
    import synth
    import paper_2404_11397_gb300 as rb

    torch.cuda.set_device(dist.local)
    device = torch.device("cuda", dist.local)
    rb.load()
    ev, data, psd = make_inputs(rb, torch, device)
    D, B = ev["geom"].shape[0], ev["n_bins"]
    event = rb.Event(ev["geom"], ev["gmst"], ev["T"], ev["f_low"], ev["f_high"], torch.view_as_complex(data), psd, B,
                     ev["theta_inj"])
    W = 4096
    theta = torch.tensor(synth.walkers("C2", W), device=device)
    logl = torch.empty(W, dtype=torch.float64, device=device)
    grad = torch.empty(W, 13, dtype=torch.float64, device=device)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=device)
    lib = rb.load()
    import ctypes

    def launch(mode, stream_handle, combined=True):
        """One step through the C ABI: rebuild the summary data from the
        event's HBM-resident strain and PSD, then log L + gradient for the
        batch -- in one call (the walkers' set-up overlapped with the summary
        sums) or as the two calls in sequence."""
        m = rb.MODES[mode]
        th, lo, gr = (ctypes.c_void_p(t.data_ptr()) for t in (theta, logl, grad))
        if combined:
            rc = lib.rb_rebuild_loglike_grad(event.handle, th, W, lo, gr, m, stream_handle)
        else:
            rc = lib.rb_event_rebuild(event.handle, None, None, None, 0, m, stream_handle)
            if rc == 0:
                rc = lib.rb_loglike_grad_batch(event.handle, th, W, lo, gr, m, stream_handle)
        if rc != 0:
            raise RuntimeError(lib.rb_last_error().decode())

    def step(mode, combined=True):
        launch(mode, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream), combined)

    graphs = {}

    def graph_for(mode, combined=True):
        """The step captured once as a CUDA graph (removes per-launch host cost)."""
        if (mode, combined) not in graphs:
            side = torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                for _ in range(3):
                    step(mode, combined)
            torch.cuda.current_stream().wait_stream(side)
            torch.cuda.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, capture_error_mode="relaxed"):
                step(mode, combined)
            torch.cuda.synchronize()
            graphs[(mode, combined)] = g
        return graphs[(mode, combined)]

    def timed(mode, K, Wm, combined=True):
        g = graph_for(mode, combined)
        for _ in range(Wm):
            g.replay()
        torch.cuda.synchronize()
        starts = [torch.cuda.Event(enable_timing=True) for _ in range(K)]
        ends = [torch.cuda.Event(enable_timing=True) for _ in range(K)]
        dist.barrier()
        torch.cuda.synchronize()
        launches0 = rb.kernel_launch_count()
        for k in range(K):
            flush.zero_()
            starts[k].record()
            g.replay()
            ends[k].record()
        torch.cuda.synchronize()
        dist.barrier()
        # kernels per step, counted from one plain (non-graph) launch of the same step
        n0 = rb.kernel_launch_count()
        step(mode, combined)
        torch.cuda.synchronize()
        per_step = rb.kernel_launch_count() - n0
        step_ms = [a.elapsed_time(b) for a, b in zip(starts, ends)]
        return step_ms, per_step * K

    def main_kernel_ms(mode, K):
        """Live duration of the main likelihood kernel (trace events recorded by
        the library around it, on its launch stream)."""
        mains = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(K)]
        for a, b in mains:  # torch creates the CUDA event on first record; the library re-records it
            a.record()
            b.record()
        torch.cuda.synchronize()
        for k in range(K):
            flush.zero_()
            rb.set_trace_events(*mains[k])
            step(mode)
        rb.set_trace_events(None, None)
        torch.cuda.synchronize()
        return [a.elapsed_time(b) for a, b in mains]

    sampler = ClockSampler(dist.local)
    # warm-up (at least ~0.5 s so the clock sampler sees the GPU under load)
    for _ in range(max(3, args.warmup)):
        step(args.mode)
    sampler.start()
    t0 = time.perf_counter()
    g = graph_for(args.mode)
    while not args.profile and time.perf_counter() - t0 < 0.5:
        for _ in range(50):
            g.replay()
        torch.cuda.synchronize()
    step_ms, launches = timed(args.mode, args.steps, 0)
    clocks = sampler.stop()
    main_ms = main_kernel_ms(args.mode, max(5, min(args.steps, 50)))
    two_ms, _ = timed(args.mode, max(3, min(args.steps, 20)), 3, combined=False)
    total_s = sum(step_ms) / 1e3
    max_total_s, value = whole_job_rate(dist, total_s, W * args.steps, device)
    main_avg_s = float(np.mean(main_ms)) / 1e3
    result = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": dist.world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": max_total_s * 1e3 / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32+f32x2(phase)+f64(sums)" if args.mode == "mixed" else args.mode,
        "data": "synthetic: seeded noise (analytic aLIGO-like PSD) + TaylorF2-tidal injection; prior-box walkers",
        "config": {"workload": WORKLOAD, "detectors": D, "T_s": ev["T"], "f_low": ev["f_low"], "f_high": ev["f_high"],
                   "n_freq": ev["N"], "n_bins": B, "walkers": W, "mode": args.mode,
                   "step": "rb_rebuild_loglike_grad: summary rebuild from the HBM-resident strain + log L and "
                           "gradient of the batch (walker set-up overlapped with the summary sums), replayed as "
                           "one captured CUDA graph",
                   "l2": "flushed (256 MiB write) before every timed step", "parallelism": f"replicas{dist.world}"},
        "gpu_launches": int(launches),
        "clocks": {k: clocks[k] for k in ("sm_mhz", "sm_max_mhz", "reasons")},
        "breakdown_ms": {"step_median": float(np.median(step_ms)), "step_p99": float(np.percentile(step_ms, 99)),
                         "two_call_step_median": float(np.median(two_ms)),
                         "main_kernel_avg": main_avg_s * 1e3,
                         "batch_evals_per_s_main_kernel_only": W / main_avg_s},
        "roofline": roofline_main(W, D, B, True, main_avg_s),
    }
    if not args.no_fp64 and args.mode != "fp64":
        K64 = max(3, min(args.steps, 20))
        s64, _ = timed("fp64", K64, 2)
        m64 = main_kernel_ms("fp64", 5)
        t64, v64 = whole_job_rate(dist, sum(s64) / 1e3, W * K64, device)
        result["fp64_path"] = {"value": v64, "unit": UNIT, "ms_per_step": t64 * 1e3 / K64,
                               "main_kernel_ms": float(np.mean(m64)),
                               "speedup_of_mixed": value / v64}
    if not args.no_configs and args.mode == "mixed":
        K3 = max(3, min(args.steps, 20))
        s3, _ = timed("mixed_f64phase", K3, 2)
        m3 = main_kernel_ms("mixed_f64phase", 5)
        t3, v3 = whole_job_rate(dist, sum(s3) / 1e3, W * K3, device)
        result["f64phase_path"] = {"value": v3, "unit": UNIT, "ms_per_step": t3 * 1e3 / K3,
                                   "main_kernel_ms": float(np.mean(m3)), "mode": "mixed_f64phase",
                                   "step": "the same rb_rebuild_loglike_grad step with the phase accumulated "
                                           "in native FP64 (the rest as the mixed path)",
                                   "cost_vs_mixed": value / v3}
    if not args.no_mala:
        result["mala_step"] = run_mala(rb, torch, event, ev, W, args, dist, device, flush)
    if not args.no_full and args.mode == "mixed":
        result["full_grid"] = run_full(rb, torch, event, ev, args, dist, device, flush, value)
    if not args.no_e2e:
        result["e2e"] = run_e2e(rb, torch, event, ev, data, psd, theta, W, args, dist, device)
        result["e2e_theta_only"] = run_e2e_theta(rb, torch, event, theta, W, args, dist, device)
    if not args.no_serving and dist.rank == 0:
        try:
            result["serving"] = run_serving(rb, torch, device)
        except Exception as exc:  # report, do not hide
            result["serving"] = {"error": str(exc)[:200]}
    if not args.no_summary_build:
        result["summary_build"] = run_summary_build(rb, torch, event, ev, flush)
    event.free()
    if not args.no_configs and args.mode == "mixed":
        result["configs"] = run_configs(rb, torch, args, dist, device, flush)
        result["bins"] = run_bins(rb, torch, device)
    return result


def run_bins(rb, torch, device, W=256):
    """Relative-binning accuracy of the two bin placements at the same bin count
    on the headline event: |log L_RB - log L_full| over W posterior-scale
    walkers (RB in FP64 through rb_loglike_batch, the full likelihood through
    rb_loglike_full_batch), with each placement's epsilon."""
    import synth
    ev, data, psd = make_inputs(rb, torch, device, "C2")
    th = torch.tensor(synth.posterior_box(ev["theta_inj"], W, seed=43), device=device)
    out = {"event": "3det_T128_f20-2048 (the headline event)", "walkers": W,
           "walkers_box": "posterior scale (+-1e-5 Mc, +-1e-3 others)",
           "error": "max / median |logL_RB (FP64) - logL_full| over the walkers"}
    for B in (200, 500):
        for bins in ("pn", "agnostic"):
            e = rb.Event(ev["geom"], ev["gmst"], ev["T"], ev["f_low"], ev["f_high"], torch.view_as_complex(data), psd,
                         B, ev["theta_inj"], bins=bins)
            d = (rb.loglike(e, th, mode="fp64") - rb.loglike_full(e, th)).abs().cpu().numpy()
            out[f"{bins}_B{B}"] = {"epsilon": e.info()["epsilon"], "max_abs_err": float(d.max()),
                                   "median_abs_err": float(np.median(d))}
            e.free()
    return out


def batch_leg(rb, torch, lib, event, th, grad, mode, K, flush, dist, device):
    """rb_loglike_batch / rb_loglike_grad_batch on device buffers: one call
    captured as a CUDA graph and replayed K times after an L2 flush each (the
    summary data are not rebuilt), and the main kernel's mean duration from
    the library's trace events over 5 eager calls.  A traced call runs set-up and
    likelihood as two kernels, a small untraced batch as one
    (launches_per_call): main_kernel_ms is then a kernel that the timed call does not run."""
    import ctypes
    W = th.shape[0]
    lo = torch.empty(W, dtype=torch.float64, device=device)
    gr = torch.empty(W, 13, dtype=torch.float64, device=device)
    m = rb.MODES[mode]

    def call():
        sh = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
        if grad:
            rc = lib.rb_loglike_grad_batch(event.handle, ctypes.c_void_p(th.data_ptr()), W,
                                           ctypes.c_void_p(lo.data_ptr()), ctypes.c_void_p(gr.data_ptr()), m, sh)
        else:
            rc = lib.rb_loglike_batch(event.handle, ctypes.c_void_p(th.data_ptr()), W, ctypes.c_void_p(lo.data_ptr()),
                                      m, sh)
        if rc != 0:
            raise RuntimeError(lib.rb_last_error().decode())

    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        for _ in range(3):
            call()
        n0 = rb.kernel_launch_count()
        call()
        per_call = rb.kernel_launch_count() - n0
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="relaxed"):
        call()
    torch.cuda.synchronize()
    for _ in range(3):
        g.replay()
    starts = [torch.cuda.Event(enable_timing=True) for _ in range(K)]
    ends = [torch.cuda.Event(enable_timing=True) for _ in range(K)]
    dist.barrier()
    torch.cuda.synchronize()
    for k in range(K):
        flush.zero_()
        starts[k].record()
        g.replay()
        ends[k].record()
    torch.cuda.synchronize()
    ms = [a.elapsed_time(b) for a, b in zip(starts, ends)]
    mains = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(5)]
    for a, b in mains:
        a.record()
        b.record()
    torch.cuda.synchronize()
    for a, b in mains:
        flush.zero_()
        rb.set_trace_events(a, b)
        call()
    rb.set_trace_events(None, None)
    torch.cuda.synchronize()
    main_s = float(np.mean([a.elapsed_time(b) for a, b in mains])) / 1e3
    del g
    t, v = whole_job_rate(dist, sum(ms) / 1e3, W * K, device)
    return {"value": v, "unit": UNIT, "walkers": W, "ms_per_call": t * 1e3 / K, "launches_per_call": per_call,
            "main_kernel_ms": main_s * 1e3, "main_kernel_form": "two kernels (traced)" if per_call == 1 else "as timed",
            "mode": mode, "grad": grad}, main_s


def run_configs(rb, torch, args, dist, device, flush):
    """The other configurations the metric is stated for, each on its own
    synthetic event (the library's strain kernel injects the signal):
    * C1: 1 detector, T = 64 s, 20-1024 Hz, 100 bins, 1000 walkers in a +-1 %
      box; log L, mixed and plain FP64;
    * C3: the same event, 4096 walkers, log L + gradient;
    * C4: 3 detectors, T = 256 s, 20-2048 Hz, 1000 bins, 16384 prior draws,
      log L + gradient, as the headline step (summary rebuild + batch in one
      captured call) and as the batch alone, plus the summary build in GB/s."""
    import ctypes
    import synth
    lib = rb.load()
    out = {}
    K = max(3, min(args.steps, 10))
    ev1, data1, psd1 = make_inputs(rb, torch, device, "C1")
    e1 = rb.Event(ev1["geom"], ev1["gmst"], ev1["T"], ev1["f_low"], ev1["f_high"], torch.view_as_complex(data1), psd1,
                  ev1["n_bins"], ev1["theta_inj"])
    th1 = torch.tensor(synth.walkers("C1"), device=device)
    c1, m1 = batch_leg(rb, torch, lib, e1, th1, False, "mixed", K, flush, dist, device)
    c1f, _ = batch_leg(rb, torch, lib, e1, th1, False, "fp64", K, flush, dist, device)
    c1["roofline"] = roofline_main(th1.shape[0], 1, ev1["n_bins"], False, m1)
    c1["fp64_path"] = c1f
    c1["config"] = "1 det (H1), T=64 s, 20-1024 Hz, 100 bins, 1000 walkers (+-1 % box), log L"
    out["C1"] = c1
    th3 = torch.tensor(synth.walkers("C3"), device=device)
    c3, m3 = batch_leg(rb, torch, lib, e1, th3, True, "mixed", K, flush, dist, device)
    c3["roofline"] = roofline_main(th3.shape[0], 1, ev1["n_bins"], True, m3)
    c3["config"] = "C1's event, 4096 walkers (+-1 % box), log L + gradient"
    out["C3"] = c3
    e1.free()
    del data1, psd1
    ev4, data4, psd4 = make_inputs(rb, torch, device, "C4")
    D4, B4 = ev4["geom"].shape[0], ev4["n_bins"]
    e4 = rb.Event(ev4["geom"], ev4["gmst"], ev4["T"], ev4["f_low"], ev4["f_high"], torch.view_as_complex(data4), psd4,
                  B4, ev4["theta_inj"])
    th4 = torch.tensor(synth.walkers("C4"), device=device)
    W4 = th4.shape[0]
    c4, m4 = batch_leg(rb, torch, lib, e4, th4, True, "mixed", K, flush, dist, device)
    c4["roofline"] = roofline_main(W4, D4, B4, True, m4)
    c4["roofline"]["traffic"] = None
    # the headline step on this event: rebuild + batch in one captured call
    lo = torch.empty(W4, dtype=torch.float64, device=device)
    gr = torch.empty(W4, 13, dtype=torch.float64, device=device)

    def step4():
        sh = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
        rc = lib.rb_rebuild_loglike_grad(e4.handle, ctypes.c_void_p(th4.data_ptr()), W4, ctypes.c_void_p(lo.data_ptr()),
                                         ctypes.c_void_p(gr.data_ptr()), rb.RB_MIXED, sh)
        if rc != 0:
            raise RuntimeError(lib.rb_last_error().decode())

    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        for _ in range(3):
            step4()
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="relaxed"):
        step4()
    torch.cuda.synchronize()
    starts = [torch.cuda.Event(enable_timing=True) for _ in range(K)]
    ends = [torch.cuda.Event(enable_timing=True) for _ in range(K)]
    for k in range(K):
        flush.zero_()
        starts[k].record()
        g.replay()
        ends[k].record()
    torch.cuda.synchronize()
    del g
    t4, v4 = whole_job_rate(dist, sum(a.elapsed_time(b) for a, b in zip(starts, ends)) / 1e3, W4 * K, device)
    c4["step"] = {"value": v4, "unit": UNIT, "ms_per_step": t4 * 1e3 / K,
                  "call": "rb_rebuild_loglike_grad (summary rebuild + log L + gradient), one captured graph"}
    c4["summary_build"] = run_summary_build(rb, torch, e4, ev4, flush)
    c4["config"] = "3 det, T=256 s, 20-2048 Hz, 1000 bins, 16384 prior draws (Mc 1.42-1.46), log L + gradient"
    out["C4"] = c4
    e4.free()
    return out


def hbm_peak_gbs():
    """Measured copy bandwidth of this machine's GPUs, if recorded beside the repository."""
    try:
        with open(ROOT / "MEASURED_PEAKS.json") as f:
            v = json.load(f).get("hbm_gbs")
        return float(v) if v else None
    except (OSError, ValueError):
        return None


def run_summary_build(rb, torch, event, ev, flush, reps=10):
    """The summary-data build (Sec. II.C) from the event's HBM-resident strain
    and PSD, three ways, each timed as a whole rb_event_rebuild call after an L2
    flush (median of `reps`):
    * mixed: fiducial waveform from per-chunk Taylor coefficients in FP32,
      reading the FP32 working copy (12 B per point and detector);
    * FP64 inline: fiducial waveform generated in FP64 at every point (24 B
      read, and the waveform stored: 16 B written);
    * FP64 stored: strain, PSD and the stored waveform streamed (40 B read).
    Runs last: it leaves the FP64 sums in place."""
    import ctypes
    lib = rb.load()
    D, N = ev["geom"].shape[0], ev["N"]
    sh = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    th = np.ascontiguousarray(event.theta_ref, dtype=np.float64)
    thp = th.ctypes.data_as(ctypes.POINTER(ctypes.c_double))

    def timed(theta_ptr, mode):
        ts = []
        for i in range(reps + 2):
            flush.zero_()
            a = torch.cuda.Event(enable_timing=True)
            b = torch.cuda.Event(enable_timing=True)
            a.record()
            rc = lib.rb_event_rebuild(event.handle, theta_ptr, None, None, 0, rb.MODES[mode], sh)
            b.record()
            torch.cuda.synchronize()
            if rc != 0:
                raise RuntimeError(lib.rb_last_error().decode())
            if i >= 2:
                ts.append(a.elapsed_time(b) / 1e3)
        return float(np.median(ts))

    t_mixed = timed(None, "mixed")
    t_inline = timed(thp, "fp64")  # a theta_ref argument discards the stored waveform
    t_stored = timed(None, "fp64")
    peak = hbm_peak_gbs()
    out = {"n_freq": N, "detectors": D, "timed": "whole rb_event_rebuild call, CUDA events, L2 flushed, median"}
    for name, t, nbytes in (("mixed", t_mixed, 12 * D * N), ("fp64_inline", t_inline, 40 * D * N),
                            ("fp64_stored", t_stored, 40 * D * N)):
        gbs = nbytes / t / 1e9
        out[name] = {"ms": t * 1e3, "bytes": nbytes, "GB_s": gbs,
                     "frac_of_measured_hbm": gbs / peak if peak else None}
    return out


def run_mala(rb, torch, event, ev, W, args, dist, device, flush):
    """The MALA local step of the sampler (Sec. II.D) for W chains on this
    event: proposal, log L + gradient and the accept step fused into the
    likelihood kernel.  Chains start in a posterior-scale box in the sampling
    coordinates (cos iota, sin dec) with the GW170817 prior box (Mc extended to
    contain the injection); draws are made before the timed region; L2
    flushed before every step.  The step is timed eagerly and as a captured
    CUDA graph (each replay's draws copied into the graph's input buffers
    before its timed region); the graph replay is the reported value."""
    import synth
    th = synth.posterior_box(ev["theta_inj"], W, seed=41)
    z = th.copy()
    z[:, 9], z[:, 12] = np.cos(th[:, 9]), np.sin(th[:, 12])
    lo = np.array([1.16, 0.125, -0.05, -0.05, 0.0, 0.0, 1.0, -0.1, 0.0, -1.0, 0.0, 0.0, -1.0])
    hi = np.array([1.21, 1.0, 0.05, 0.05, 5000.0, 5000.0, 75.0, 0.1, 2 * np.pi, 1.0, np.pi, 2 * np.pi, 1.0])
    # step sizes of the order of the posterior widths of this event
    eps = np.array([1e-6, 1e-3, 5e-5, 5e-5, 5.0, 5.0, 0.1, 2e-6, 3e-3, 3e-3, 2e-3, 2e-4, 3e-4])
    zt = torch.tensor(z, device=device)
    logp, gz = rb.mala_init(event, zt, lo, hi, mode=args.mode)
    K = max(3, min(args.steps, 20))
    gen = torch.Generator(device=device).manual_seed(7)
    xi = torch.randn(K + 3, W, 13, dtype=torch.float64, device=device, generator=gen)
    u = torch.rand(K + 3, W, dtype=torch.float64, device=device, generator=gen)
    for i in range(3):
        rb.mala_step(event, zt, logp, gz, eps, lo, hi, xi[i], u[i], mode=args.mode)
    starts = [torch.cuda.Event(enable_timing=True) for _ in range(K)]
    ends = [torch.cuda.Event(enable_timing=True) for _ in range(K)]
    dist.barrier()
    torch.cuda.synchronize()
    accs = []
    for k in range(K):
        flush.zero_()
        starts[k].record()
        accs.append(rb.mala_step(event, zt, logp, gz, eps, lo, hi, xi[3 + k], u[3 + k], mode=args.mode))
        ends[k].record()
    torch.cuda.synchronize()
    eager_ms = [a.elapsed_time(b) for a, b in zip(starts, ends)]
    # the same steps replayed from one captured graph
    xi_in, u_in = xi[0].clone(), u[0].clone()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        rb.mala_step(event, zt, logp, gz, eps, lo, hi, xi_in, u_in, mode=args.mode)
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="relaxed"):
        acc_g = rb.mala_step(event, zt, logp, gz, eps, lo, hi, xi_in, u_in, mode=args.mode)
    torch.cuda.synchronize()
    dist.barrier()
    for k in range(K):
        xi_in.copy_(xi[3 + k])
        u_in.copy_(u[3 + k])
        flush.zero_()
        starts[k].record()
        g.replay()
        ends[k].record()
        accs.append(acc_g.float().mean())
    torch.cuda.synchronize()
    acc = float(torch.stack([a.float().mean() for a in accs]).mean().item())
    ms = [a.elapsed_time(b) for a, b in zip(starts, ends)]
    del g
    t, v = whole_job_rate(dist, sum(ms) / 1e3, W * K, device)
    return {"value": v, "unit": "chain-steps/s", "chains": W, "steps": 2 * K, "ms_per_step": t * 1e3 / K,
            "eager_ms_per_step": float(np.mean(eager_ms)), "acceptance": acc, "mode": args.mode,
            "step": "rb_mala_step: proposal kernel, set-up, log L + adjoint with the accept step fused; "
                    "value from K replays of the step captured as one CUDA graph, after K eager steps"}


def run_full(rb, torch, event, ev, args, dist, device, flush, rb_value, W=1024):
    """The full-grid (un-binned) log-likelihood of the same event for W prior
    draws: the quantity relative binning replaces (Sec. II.C), every grid
    point of every detector evaluated per walker.  L2 flushed before every
    call."""
    import synth
    th = torch.tensor(synth.walkers("C2", W), device=device)
    K = max(3, min(args.steps, 10))
    for _ in range(3):
        rb.loglike_full(event, th)
    starts = [torch.cuda.Event(enable_timing=True) for _ in range(K)]
    ends = [torch.cuda.Event(enable_timing=True) for _ in range(K)]
    dist.barrier()
    torch.cuda.synchronize()
    for k in range(K):
        flush.zero_()
        starts[k].record()
        rb.loglike_full(event, th)
        ends[k].record()
    torch.cuda.synchronize()
    ms = [a.elapsed_time(b) for a, b in zip(starts, ends)]
    t, v = whole_job_rate(dist, sum(ms) / 1e3, W * K, device)
    N = ev["N"]
    achieved = FULL_FLOPS_PER_WALKER_POINT * v * N / 1e12
    peak = fp32_peak_tflops()
    return {"value": v, "unit": "full-grid evals/s", "walkers": W, "calls": K, "ms_per_call": t * 1e3 / K,
            "grid_points_per_eval": int(N * ev["geom"].shape[0]), "walker_points_per_s": v * N,
            "rb_speedup": rb_value / v,
            "roofline": {"bound": "alu", "kernel": "k_full_z (fp32 pipe)", "achieved": achieved, "peak": peak,
                         "unit": "TFLOP/s", "frac": achieved / peak,
                         "flops_per_walker_point": FULL_FLOPS_PER_WALKER_POINT,
                         "peak_source": "derived: 152 SMs x 128 FP32 lanes x 2 flop x 2070 MHz"},
            "call": "rb_loglike_full_batch: set-up, per-walker grid sum, combination"}


def run_e2e(rb, torch, event, ev, data, psd, theta, W, args, dist, device):
    """Same metric through the public API on pinned host buffers
    (rb_rebuild_loglike_grad_host): strain/PSD and walkers brought in every
    step (strain/PSD read by a kernel over the host link, walkers copied), log
    L and gradient written back to the pinned outputs, the stream
    synchronised."""
    import ctypes
    D, N = ev["geom"].shape[0], ev["N"]
    h_data = [data[d].cpu().pin_memory() for d in range(D)]
    h_psd = [psd[d].cpu().pin_memory() for d in range(D)]
    h_theta = theta.cpu().pin_memory()
    h_logl = torch.empty(W, dtype=torch.float64).pin_memory()
    h_grad = torch.empty(W, 13, dtype=torch.float64).pin_memory()
    lib = rb.load()
    dp = (ctypes.c_void_p * D)(*[t.data_ptr() for t in h_data])
    pp = (ctypes.c_void_p * D)(*[t.data_ptr() for t in h_psd])
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)

    def step():
        rc = lib.rb_rebuild_loglike_grad_host(event.handle, dp, pp, ctypes.c_void_p(h_theta.data_ptr()), W,
                                              ctypes.c_void_p(h_logl.data_ptr()), ctypes.c_void_p(h_grad.data_ptr()),
                                              rb.MODES[args.mode], stream)
        if rc != 0:
            raise RuntimeError(lib.rb_last_error().decode())

    for _ in range(max(3, args.warmup)):
        step()
    K = args.steps
    dist.barrier()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(K):
        step()
    torch.cuda.synchronize()
    el, ev_rate = whole_job_rate(dist, time.perf_counter() - t0, W * K, device)
    return {"value": ev_rate, "unit": UNIT, "ms_per_step": el * 1e3 / K,
            "h2d_bytes_per_step": int(D * N * 3 * 8 + W * 13 * 8), "d2h_bytes_per_step": int(W * 14 * 8)}


def run_e2e_theta(rb, torch, event, theta, W, args, dist, device):
    """The sampler's form of the end-to-end call (rb_loglike_grad_host): the
    event's data stay resident; each step copies the walkers in from pinned
    host memory and writes log L and the gradient to pinned host outputs, then
    synchronises.  No summary rebuild."""
    import ctypes
    h_theta = theta.cpu().pin_memory()
    h_logl = torch.empty(W, dtype=torch.float64).pin_memory()
    h_grad = torch.empty(W, 13, dtype=torch.float64).pin_memory()
    lib = rb.load()
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)

    def step():
        rc = lib.rb_loglike_grad_host(event.handle, ctypes.c_void_p(h_theta.data_ptr()), W,
                                      ctypes.c_void_p(h_logl.data_ptr()), ctypes.c_void_p(h_grad.data_ptr()),
                                      rb.MODES[args.mode], stream)
        if rc != 0:
            raise RuntimeError(lib.rb_last_error().decode())

    for _ in range(max(3, args.warmup)):
        step()
    K = args.steps
    dist.barrier()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(K):
        step()
    torch.cuda.synchronize()
    el, rate = whole_job_rate(dist, time.perf_counter() - t0, W * K, device)
    return {"value": rate, "unit": UNIT, "ms_per_step": el * 1e3 / K, "h2d_bytes_per_step": int(W * 13 * 8),
            "d2h_bytes_per_step": int(W * 14 * 8),
            "call": "rb_loglike_grad_host: walkers in, log L + gradient out, event resident (no rebuild)"}


def run_serving(rb, torch, device, loads=(0.5, 0.8, 0.95), seconds: float = 2.0, n_events: int = 64):
    """Continuous-batching serving loop over n_events resident synthetic events
    (T uniform in {64, 128, 256} s, 2 or 3 detectors, 100-1000 bins), each
    request 256-8192 walkers with the gradient.  Saturation: four client
    threads keep 32 requests queued for 3 s.  Then Poisson arrivals at each
    fraction of saturation in `loads` for `seconds` each.  Latency p50/p99: the
    server's own measurement, rb_submit to results in host memory;
    client_p50/p99: submit to the poll's return in this Python client (its
    thread hand-offs included)."""
    import synth
    rng = np.random.default_rng(20240417)
    site_sets = [("H1", "L1"), ("H1", "V1"), ("L1", "V1"), ("H1", "L1", "V1")]
    base = {}
    events = []
    for i in range(n_events):
        T = float(rng.choice([64.0, 128.0, 256.0]))
        sites = site_sets[int(rng.integers(0, len(site_sets)))]
        B = int(rng.integers(100, 1001))
        key = (T, sites)
        if key not in base:  # noise and PSD per (duration, detector set); signals differ per event
            ev = synth.make_event("C2", T=T, sites=sites)
            noise = torch.tensor(np.stack([ev["noise"].real, ev["noise"].imag], -1), device=device)
            base[key] = (ev, noise, torch.tensor(ev["psd"], device=device))
        ev, noise, psd = base[key]
        th_inj = ev["theta_inj"].copy()
        th_inj[0] *= 1.0 + 0.01 * (rng.random() - 0.5)  # a different source per event
        th_inj[6] = 30.0 + 20.0 * rng.random()
        D, N = ev["geom"].shape[0], ev["N"]
        data = torch.empty(D, N, 2, dtype=torch.float64, device=device)
        for d in range(D):
            h = rb.strain(ev["geom"][d], ev["gmst"], th_inj, ev["T"], ev["kmin"], N, device=device)
            data[d] = noise[d] + torch.view_as_real(h)
        events.append(rb.Event(ev["geom"], ev["gmst"], T, ev["f_low"], ev["f_high"], torch.view_as_complex(data), psd,
                               B, th_inj))
        del data
    pool = synth.walkers("C2", 8192)
    srv = rb.Server(hbm_budget_bytes=4 << 30, max_slots=8, max_walkers=8192, mode="mixed")
    for i in range(len(events)):  # warm-up: every event once
        t = srv.submit(events[i], pool[:256], want_grad=True)
        srv.poll(t, timeout_us=-1)
    sizes = rng.integers(256, 8193, 4000)
    mean_w = float(np.mean(sizes))
    # saturation throughput: 4 client threads keep 32 requests queued for ~3 s
    # (one Python client thread cannot submit and collect fast enough); they
    # call rb_submit / rb_poll directly with preallocated output buffers
    import ctypes
    lib = rb.load()
    pool_p = pool.ctypes.data
    n_cli = 4
    done = [0] * n_cli

    def submit_raw(ev, W):
        t = ctypes.c_uint64()
        rc = lib.rb_submit(srv._h, ev.handle, ctypes.cast(pool_p, rb._lib.c_double_p), W, 1, ctypes.byref(t))
        if rc != 0:
            raise RuntimeError(lib.rb_last_error().decode())
        return t.value

    def poll_raw(t, out_l, out_g):
        rc = lib.rb_poll(srv._h, t, -1, out_l.ctypes.data_as(rb._lib.c_double_p), out_g.ctypes.data_as(rb._lib.c_double_p))
        if rc != 0:
            raise RuntimeError(lib.rb_last_error().decode())

    def client(ci):
        inflight, k = [], ci
        out_l, out_g = np.empty(8192), np.empty((8192, 13))
        t_end = time.perf_counter() + 3.0
        while time.perf_counter() < t_end:
            while len(inflight) < 32 // n_cli:
                W = int(sizes[k % len(sizes)])
                inflight.append((submit_raw(events[k % len(events)], W), W))
                k += n_cli
            t, W = inflight.pop(0)
            poll_raw(t, out_l, out_g)
            done[ci] += W
        for t, W in inflight:
            poll_raw(t, out_l, out_g)
            done[ci] += W

    tick = time.perf_counter()
    cl = [threading.Thread(target=client, args=(i,)) for i in range(n_cli)]
    for c in cl:
        c.start()
    for c in cl:
        c.join()
    sat = sum(done) / (time.perf_counter() - tick)
    s0 = srv.stats()
    srv.latency(reset=True)
    points = []
    import queue
    for load in loads:
        rate = load * sat / mean_w  # requests per second
        lat = []
        tickets = queue.Queue()

        def collector():
            out_l, out_g = np.empty(8192), np.empty((8192, 13))
            while True:
                item = tickets.get()
                if item is None:
                    return
                t, t0 = item
                poll_raw(t, out_l, out_g)
                lat.append(time.perf_counter() - t0)

        cols = [threading.Thread(target=collector, daemon=True) for _ in range(2)]
        for c in cols:
            c.start()
        n_sub = 2  # two independent Poisson streams at rate / 2 each: one Poisson stream at `rate`
        counts = [[0, 0] for _ in range(n_sub)]
        t_start = time.perf_counter()
        t_end = t_start + seconds

        def submitter(si):
            r = np.random.default_rng(1000 * si + int(load * 100))
            nxt = t_start
            while nxt < t_end:
                now = time.perf_counter()
                if now < nxt:
                    time.sleep(min(nxt - now, 1e-3))
                    continue
                W = int(r.integers(256, 8193))
                i = int(r.integers(0, len(events)))
                t0 = time.perf_counter()
                tickets.put((submit_raw(events[i], W), t0))
                counts[si][0] += 1
                counts[si][1] += W
                nxt += r.exponential(n_sub / rate)

        subs = [threading.Thread(target=submitter, args=(i,)) for i in range(n_sub)]
        for x in subs:
            x.start()
        for x in subs:
            x.join()
        n_req = sum(c[0] for c in counts)
        walkers = sum(c[1] for c in counts)
        for _ in cols:
            tickets.put(None)
        for c in cols:
            c.join(timeout=30)
        elapsed = time.perf_counter() - t_start
        lat_ms = np.array(lat) * 1e3
        server = srv.latency(reset=True)
        tot = server["total"]
        points.append({"offered_load": load, "requests": n_req, "throughput_evals_s": walkers / elapsed,
                       "p50_ms": tot["p50_ms"], "p99_ms": tot["p99_ms"], "max_ms": tot["max_ms"],
                       "client_p50_ms": float(np.percentile(lat_ms, 50)),
                       "client_p99_ms": float(np.percentile(lat_ms, 99)),
                       "parts_p99_ms": {k: server[k]["p99_ms"] for k in ("queue", "issue", "device")},
                       "parts_max_ms": {k: server[k]["max_ms"] for k in ("queue", "issue", "device")}})
    stats = srv.stats()
    srv.close()
    for e in events:
        e.free()
    launches = stats["graph_launches"] + stats["plain_launches"]
    return {"events": len(events), "request_walkers": "uniform 256-8192, with gradient",
            "saturation_evals_s": sat, "loads": points,
            "requests_per_launch": stats["completed"] / max(1, launches),
            "padding_fraction": stats["walkers_run"] / max(1, stats["walkers_requested"]) - 1.0,
            "launches": int(launches), "graph_instantiations": int(stats["graphs_captured"]),
            "graph_updates": int(stats["graph_updates"]), "max_in_flight": int(stats["max_in_flight"]),
            "saturation_requests_per_launch": (s0["completed"]) / max(1, s0["graph_launches"] + s0["plain_launches"])}


# ---------------------------------------------------------------------------
def oracle_step_estimate(target_s: float = 12.0):
    """Time the FP64 CPU oracle on a bounded sample of the same workload: the
    full summary build plus log L + gradient of S walkers; returns the
    per-step time extrapolated to 4096 walkers."""
    import oracle
    import synth
    ev = synth.make_event("C2")
    ev["data"] = ev["noise"] + np.stack([oracle.strain(ev["theta_inj"], ev["geom"][d], ev["gmst"], ev["f"])
                                         for d in range(ev["geom"].shape[0])])
    threads = oracle.default_threads()
    t0 = time.perf_counter()
    edges = oracle.bin_edges(ev, ev["n_bins"])
    s = oracle.summary(ev, ev["theta_inj"], edges)
    t_sum = time.perf_counter() - t0
    th = synth.walkers("C2", 4096)
    t0 = time.perf_counter()
    oracle.loglike_rb(ev, s, th[:threads * 2], grad=True, nthreads=threads)
    t_probe = (time.perf_counter() - t0) / (threads * 2)
    S = int(max(threads * 2, min(4096, (target_s - t_sum) / max(t_probe, 1e-6))))
    t0 = time.perf_counter()
    oracle.loglike_rb(ev, s, th[:S], grad=True, nthreads=threads)
    t_walk = (time.perf_counter() - t0) / S
    step_s = t_sum + 4096 * t_walk
    # one core: the summary build is single-threaded already; walkers on one thread
    S1 = 32
    t0 = time.perf_counter()
    oracle.loglike_rb(ev, s, th[:S1], grad=True, nthreads=1)
    t_walk1 = (time.perf_counter() - t0) / S1
    return {"step_s": step_s, "step_s_1core": t_sum + 4096 * t_walk1, "cores": threads,
            "sample": f"summary build (full) + logL+grad of {S} of 4096 walkers, extrapolated to 4096 "
                      f"(summary {t_sum:.2f} s, {t_walk * 1e3:.3f} ms/walker on {threads} threads; "
                      f"{t_walk1 * 1e3:.3f} ms/walker on 1 thread from {S1} walkers)"}


def run_reference(args, dist: Dist):
    if dist.rank != 0:
        return None
    steps = []
    # warm-up steps (smaller bounded samples: the oracle keeps no state
    # between steps, but its library, caches and thread pool warm up), then
    # at most 3 timed steps so that the run stays within about a minute
    Wu = max(3, args.warmup)
    for _ in range(Wu):
        oracle_step_estimate(target_s=1.5)
    K = max(1, min(args.steps, 3))
    info = None
    for _ in range(K):
        info = oracle_step_estimate(target_s=8.0)
        steps.append(info["step_s"])
    value = 4096 / float(np.mean(steps))
    return {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": dist.world, "steps": K, "warmup": Wu,
            "ms_per_step": float(np.mean(steps)) * 1e3, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic", "impl": "reference",
            "config": {"workload": WORKLOAD, "detectors": 3, "n_bins": 500, "walkers": 4096},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": info["cores"], "kind": "oracle",
                             "sample": info["sample"], "value_1_core": 4096 / info["step_s_1core"]},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}


def main():
    args = parse()
    if args.profile:
        args.no_e2e = args.no_cpu = args.no_serving = args.no_fp64 = args.no_mala = args.no_full = True
        args.no_summary_build = args.no_configs = True
    dist = Dist()
    if args.impl == "reference":
        dist.init("gloo")
        res = run_reference(args, dist)
        if res is not None:
            print(json.dumps(res), flush=True)
        dist.close()
        return 0
    import torch
    dist.init("nccl" if torch.cuda.is_available() else "gloo")
    res = run_gb300(args, dist)
    if dist.rank == 0:
        if not args.no_cpu and dist.world == 1:
            est = oracle_step_estimate()
            res["cpu_baseline"] = {"value": 4096 / est["step_s"], "unit": UNIT, "cores": est["cores"],
                                   "kind": "oracle", "sample": est["sample"],
                                   "value_1_core": 4096 / est["step_s_1core"]}
        print(json.dumps(res), flush=True)
    dist.close()
    return 0


if __name__ == "__main__":
    sys.exit(main())
