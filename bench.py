#!/usr/bin/env python3
"""Throughput of the batched FP32 TWA ensemble on one GB300 (and replicas on N GPUs).

Workload: 3D Gaussian-random-field condensation (Sec. IV.B, Eq. kspaceGauss) on a
128^3 periodic grid, 256 sampled streams plus the classical field, FP32 fields,
kick-drift-kick steps at dt from the pi/4 kinetic rule, ensemble moments (FP64
accumulation, per-mode occupations included) every 10 steps.  One bench step is
one output interval: 10 KDK steps of the whole batch plus its moments, through
the public call twa_advance on device-resident inputs.  Metric: TWA
cell-updates/s = streams x cells x KDK steps / s (the classical field is
evolved too but not counted).

Also reported: the dominant pass's achieved HBM bandwidth (algorithmic bytes /
CUDA-event time of its launches in the timed region) against the measured copy
bandwidth; the FP64 CPU oracle on this host's cores (cpu_baseline); the plain
FP64 single-realization GPU path and a cuFFT/torch reference step (context);
end-to-end throughput of twa_run with host buffers.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl twa|reference]
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "TWA cell-updates/s, FP32 batched vs FP64 plain on 1 GB300, at stated err; %HBM peak"
UNIT = "cell-updates/s"
GRID_M = 128
STREAMS = 256
OUT_EVERY = 10
SEED = 2024


def _args():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["twa", "reference"], default="twa")
    ap.add_argument("--no-extras", action="store_true", help="skip cpu/f64/cufft/e2e side measurements")
    ap.add_argument("--streams", type=int, default=STREAMS, help="streams per batch (smaller batches for ncu captures)")
    ap.add_argument("--no-tune", action="store_true", help="skip the autotuner (default pass shapes, axis pipeline)")
    ap.add_argument("--paper-scale", action="store_true",
                    help="only measure the 512^3 x 64-stream soliton (about 175 GB on the device) and print it")
    return ap.parse_args()


def _peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        d = json.load(open(p))
        return float(d["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


def _cores():
    try:
        return len(os.sched_getaffinity(0))
    except AttributeError:
        return os.cpu_count() or 1


# ------------------------------------------------------------------------------------------
class ClockSampler:
    """nvidia-smi clock / throttle-reason samples taken while the timed region runs."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.path = None

    def __enter__(self):
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.gpu}", f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except (OSError, FileNotFoundError):
            self.proc = None
        return self

    def __exit__(self, *a):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        if self.proc is None or not self.path or not os.path.exists(self.path):
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        sm, smax, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            f = [x.strip() for x in line.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                smax = float(f[2])
            except ValueError:
                continue
            for n, v in zip(names, f[5:9]):
                if v.lower() == "active":
                    reasons.add(n)
        os.unlink(self.path)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": smax,
                "reasons": sorted(reasons), "samples": len(sm)}


# ------------------------------------------------------------------------------------------
def _workload(streams=STREAMS):
    import twa_inputs as ti
    return ti.workload_3d_condensation(GRID_M, streams, 2000)


def _oracle_rate(w, n_fields=2, budget_s=12.0):
    """FP64 oracle (scipy.fft on all host cores) on a bounded sample of the workload."""
    import numpy as np
    from oracle import sp, twa
    cl = w.psi_cl()
    b = twa.sample(cl, w.noise_seed, n_fields, w.phys.n_tot, w.grid.dV)[1:]
    sp.step(b, w.phys.hbar_m, w.phys.C, w.phys.dt, 1.0, 3)          # warm the FFT plans
    t0 = time.perf_counter()
    n = 0
    while True:
        b = sp.step(b, w.phys.hbar_m, w.phys.C, w.phys.dt, 1.0, 3)
        n += 1
        el = time.perf_counter() - t0
        if el > budget_s or n >= 50:
            break
    return n_fields * w.grid.cells * n / el, n, el


def run_reference(args):
    """Reference arm: the FP64 oracle as it stands, timed on this host's cores."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    import numpy as np
    from oracle import sp, twa
    w = _workload()
    cl = w.psi_cl()
    nf = 2
    b = twa.sample(cl, w.noise_seed, nf, w.phys.n_tot, w.grid.dV)[1:]
    for _ in range(args.warmup):
        b = sp.step(b, w.phys.hbar_m, w.phys.C, w.phys.dt, 1.0, 3)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        b = sp.step(b, w.phys.hbar_m, w.phys.C, w.phys.dt, 1.0, 3)
    el = time.perf_counter() - t0
    val = nf * w.grid.cells * args.steps / el
    sample = f"{nf} sampled streams of the 128^3 workload, 1 KDK step per bench step (FP64 numpy/scipy, workers={sp.WORKERS})"
    line = {
        "impl": "reference", "metric": METRIC, "value": val, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * el / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": "3D Gaussian-random-field condensation 128^3 (oracle sample)", "streams": nf},
        "cpu_baseline": {"value": val, "unit": UNIT, "cores": _cores(), "kind": "oracle", "sample": sample},
        "e2e": {"value": val, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


def _f64_plain_rate(w, steps=2):
    import torch
    from paper_2310_07119_gb300 import Ensemble, F64_PLAIN
    ens = Ensemble([w.grid], w.phys.hbar_m, w.phys.C, w.phys.dt, w.phys.n_tot, [1], precision=F64_PLAIN,
                   want_modes=False)
    ens.sample([w.psi_cl()], w.noise_seed)
    ens.step(1)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    ens.step(steps)
    e1.record()
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1)
    ens.close()
    fields = 2  # the classical field and the stream
    return fields * w.grid.cells * steps / (ms * 1e-3)


def _cufft_reference_rate(w, batch=32, steps=5):
    """One KDK step written with torch.fft (cuFFT) and torch elementwise ops (timing reference only)."""
    import torch
    dev = torch.device("cuda")
    m = w.grid.n[0]
    k = 2 * math.pi * torch.fft.fftfreq(m, d=1.0 / m, dtype=torch.float64)
    k2 = (k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :] ** 2).to(dev)
    kin = torch.exp(-1j * torch.remainder(w.phys.hbar_m * k2 * w.phys.dt / 2, 2 * math.pi)).to(torch.complex64)
    inv = torch.where(k2 > 0, -w.phys.C / k2, torch.zeros_like(k2)).to(torch.float32)
    psi = torch.randn((batch, m, m, m), dtype=torch.complex64, device=dev)
    kick = w.phys.dt / (2 * w.phys.hbar_m)

    def step(p):
        V = torch.fft.ifftn(torch.fft.fftn(p.abs() ** 2, dim=(1, 2, 3)) * inv, dim=(1, 2, 3)).real
        p = p * torch.exp(-1j * kick * V)
        p = torch.fft.ifftn(torch.fft.fftn(p, dim=(1, 2, 3)) * kin, dim=(1, 2, 3))
        V = torch.fft.ifftn(torch.fft.fftn(p.abs() ** 2, dim=(1, 2, 3)) * inv, dim=(1, 2, 3)).real
        return p * torch.exp(-1j * kick * V)

    psi = step(psi)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(steps):
        psi = step(psi)
    e1.record()
    torch.cuda.synchronize()
    return batch * m ** 3 * steps / (e0.elapsed_time(e1) * 1e-3)


def _adaptive_rate(ens, w, n_out=3, c_f=0.01):
    """The bench batch advanced with the dynamic time step of Sec. III.B.2 (twa_advance_adaptive):
    the step is chosen before every output interval, which reads max|V| back (one host
    synchronization per interval) and runs the interval without graph replay."""
    import torch
    from paper_2310_07119_gb300 import twa_advance_adaptive
    ens.sample([w.psi_cl()], w.noise_seed)
    twa_advance_adaptive(ens.h, ens.psi, 1, OUT_EVERY, c_f, ens.new_series(OUT_EVERY, OUT_EVERY))
    series = ens.new_series(n_out * OUT_EVERY, OUT_EVERY)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    times = twa_advance_adaptive(ens.h, ens.psi, n_out, OUT_EVERY, c_f, series)
    e1.record()
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1)
    steps = (times[1:] - times[:-1]) / OUT_EVERY
    return {"value": STREAMS * w.grid.cells * OUT_EVERY * n_out / (ms * 1e-3), "unit": UNIT,
            "ms_per_step": ms / n_out, "c_f": c_f, "dt_first": float(steps[0]), "dt_last": float(steps[-1])}


def _phase_moments_cost(ens, w, reps=3):
    """Amplitude and phase variances (Eq. varA, Eq. varPhi) of the bench batch: two reads of every
    stream per call (means, then deviations and phases)."""
    import torch
    from paper_2310_07119_gb300 import twa_phase_moments
    tot = twa_phase_moments(ens.h, 0, ens.psi)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(reps):
        twa_phase_moments(ens.h, 0, ens.psi, totals=tot)
    e1.record()
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / reps
    nbytes = 2 * STREAMS * w.grid.cells * 8
    return {"ms_per_call": ms, "GBps": nbytes / (ms * 1e-3) / 1e9, "var_a": float(tot[0]), "var_phi": float(tot[1])}


def _observable_cost(ens, w, reps=3):
    """Stream averages of user functions (Appendix B's synthesizer) on the bench batch: one read of
    every stream per call, f evaluated and summed in FP64, or in FP32 with float-pair sums.  A
    polynomial and a transcendental f."""
    import torch
    from paper_2310_07119_gb300 import Observable
    out = {}
    nbytes = (STREAMS + 1) * w.grid.cells * 8
    for name, (fre, fim, fp32) in {"density": ("re*re + im*im", None, False),
                                   "phase_and_amplitude": ("atan2(im, re)", "sqrt(re*re + im*im)", False),
                                   "density_fp32": ("re*re + im*im", None, True),
                                   "phase_and_amplitude_fp32": ("atan2(im, re)", "sqrt(re*re + im*im)", True)}.items():
        ob = Observable(fre, fim, fp32=fp32)
        r = ob(ens)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(reps):
            ob(ens)
        e1.record()
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1) / reps
        out[name] = {"ms_per_call": ms, "GBps": nbytes / (ms * 1e-3) / 1e9, "total_re": r["total"].real}
        ob.close()
    return out


def _particles_rate(ens, w, n_out=3):
    """The bench batch advanced with one test particle per stream (Sec. III.D): the particle update
    runs before every step, with the Poisson field brought to real space where the pipeline keeps
    it spectral.  Reports the rate and the particles' spread after the timed interval."""
    import numpy as np
    import torch
    from paper_2310_07119_gb300 import twa_advance, twa_particles_get, twa_particles_set
    ns = STREAMS + 1
    r0 = np.tile([0.5, 0.5, 0.5], (ns, 1))
    ens.sample([w.psi_cl()], w.noise_seed)
    twa_particles_set(ens.h, 0, r0, np.zeros((ns, 3)))
    twa_advance(ens.h, ens.psi, OUT_EVERY, OUT_EVERY, ens.new_series(OUT_EVERY, OUT_EVERY))
    series = ens.new_series(n_out * OUT_EVERY, OUT_EVERY)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    twa_advance(ens.h, ens.psi, n_out * OUT_EVERY, OUT_EVERY, series)
    e1.record()
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1)
    r, p = twa_particles_get(ens.h, 0, ns, 3)
    d = np.mod(r[1:] - r[0] + 0.5, 1.0) - 0.5
    return {"value": STREAMS * w.grid.cells * OUT_EVERY * n_out / (ms * 1e-3), "unit": UNIT, "ms_per_step": ms / n_out,
            "spread_x": float(np.sqrt(np.mean(np.sum((d - d.mean(0)) ** 2, 1)))),
            "spread_p": float(np.sqrt(np.mean(np.sum((p[1:] - p[1:].mean(0)) ** 2, 1))))}


def _one_d_rate():
    """The 1D workload (256 cells, 32 streams + classical, 1000 KDK steps, moments every 10): the
    whole run in one on-chip launch and a finishing one on the FP32 path; the FP64 path on the same run."""
    import torch
    import twa_inputs as ti
    from paper_2310_07119_gb300 import Ensemble, F32, F64_PLAIN, twa_advance
    w = ti.workload_1d_bump(256, 32, 1000)
    out = {}
    for name, prec in (("f32", F32), ("f64_plain", F64_PLAIN)):
        ens = Ensemble([w.grid], w.phys.hbar_m, w.phys.C, w.phys.dt, w.phys.n_tot, [w.n_real], precision=prec)
        ens.sample([w.psi_cl()], w.noise_seed)
        twa_advance(ens.h, ens.psi, 100, w.out_every, ens.new_series(100, w.out_every))
        series = ens.new_series(w.n_steps, w.out_every)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        twa_advance(ens.h, ens.psi, w.n_steps, w.out_every, series)
        e1.record()
        torch.cuda.synchronize()
        out[name] = w.n_real * w.grid.cells * w.n_steps / (e0.elapsed_time(e1) * 1e-3)
        ens.close()
    return {"value": out["f32"], "f64_plain": out["f64_plain"], "unit": UNIT,
            "workload": "1D Gaussian bump 256 cells x 32 streams, 1000 KDK steps, moments every 10 (whole run on chip: instruction latency)"}


def _uneven_rate(steps=3):
    """Uneven multi-instance batch in one handle (2D two-soliton merger: 512^2 x 128, 1024^2 x 64 and
    2048^2 x 16 streams), moments every 10 steps: the tuned batch mode, then each mode (one instance
    after another, parallel graph branches, one persistent launch per interval) and each instance in
    a handle of its own (the sum of the parts)."""
    import torch
    import twa_inputs as ti
    from paper_2310_07119_gb300 import (BATCH_FORK, BATCH_PERSISTENT, BATCH_SERIAL, Ensemble, twa_advance,
                                        twa_get_batch_mode, twa_set_batch_mode)
    ws = [ti.workload_2d_merger(m, nr, 1000) for m, nr in ((512, 128), (1024, 64), (2048, 16))]
    p = ws[0].phys

    def timed(ens):
        ens.sample([w.psi_cl() for w in ws] if len(ens.grids) == len(ws) else [ens._w.psi_cl()], SEED)
        twa_advance(ens.h, ens.psi, 2 * OUT_EVERY, OUT_EVERY, ens.new_series(2 * OUT_EVERY, OUT_EVERY))
        series = ens.new_series(steps * OUT_EVERY, OUT_EVERY)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        twa_advance(ens.h, ens.psi, steps * OUT_EVERY, OUT_EVERY, series)
        e1.record()
        torch.cuda.synchronize()
        return e0.elapsed_time(e1) / steps

    ens = Ensemble([w.grid for w in ws], p.hbar_m, p.C, p.dt, p.n_tot, [w.n_real for w in ws], want_modes=True)
    ens.autotune(_tune_cache_path(torch.cuda.current_device()))
    tuned = twa_get_batch_mode(ens.h)
    ms = timed(ens)
    modes = {}
    for name, m in (("serial", BATCH_SERIAL), ("fork", BATCH_FORK), ("persistent", BATCH_PERSISTENT)):
        twa_set_batch_mode(ens.h, m)
        modes[name] = timed(ens)
    ens.close()
    alone = []
    for w in ws:
        e = Ensemble([w.grid], p.hbar_m, p.C, p.dt, p.n_tot, [w.n_real], want_modes=True)
        e._w = w
        e.autotune(_tune_cache_path(torch.cuda.current_device()))
        alone.append(timed(e))
        e.close()
    cu = sum(w.n_real * w.grid.cells for w in ws) * OUT_EVERY
    return {"value": cu * steps / (ms * steps * 1e-3), "unit": UNIT, "ms_per_step": ms,
            "tuned_mode": ["serial", "fork", "persistent"][tuned],
            "ms_per_step_by_mode": modes, "ms_per_step_instances_alone": alone,
            "ms_per_step_sum_of_parts": sum(alone),
            "workload": "2D two-soliton merger 512^2 x 128 + 1024^2 x 64 + 2048^2 x 16 streams in one handle, "
                        f"{OUT_EVERY} KDK steps + moments per step, batch {sum((w.n_real + 1) * w.grid.cells for w in ws) * 8 / 1e9:.2f} GB"}


def _e2e(ens, w, steps=2, n_run=50):
    """twa_run from a pinned host psi_cl, then the final moments a user reads (<rho>, <n_k>, Var n_k)
    and the scalar series back to pinned host memory; all copies inside the timed region."""
    import torch
    from paper_2310_07119_gb300 import twa_moments, twa_run
    cl_host = torch.from_numpy(w.psi_cl().reshape(-1)).pin_memory()
    cl_dev = torch.empty_like(cl_host, device=ens.device)
    series = ens.new_series(n_run, OUT_EVERY)
    series_host = torch.empty(series.shape, dtype=series.dtype).pin_memory()
    cells = w.grid.cells
    outs = {k: torch.empty(cells, dtype=torch.float64, device=ens.device) for k in ("rho_mean", "nk_mean", "nk_var")}
    hosts = {k: torch.empty(cells, dtype=torch.float64).pin_memory() for k in outs}
    st = torch.cuda.current_stream()

    def one():
        cl_dev.copy_(cl_host, non_blocking=True)
        twa_run(ens.h, cl_dev, SEED, n_run, OUT_EVERY, ens.psi, series)
        twa_moments(ens.h, 0, ens.psi, outs)
        series_host.copy_(series, non_blocking=True)
        for k in outs:
            hosts[k].copy_(outs[k], non_blocking=True)

    one()                                  # warm-up (graph capture happens here)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(st)
    for _ in range(steps):
        one()
    e1.record(st)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1)
    val = STREAMS * w.grid.cells * n_run * steps / (ms * 1e-3)
    d2h = series_host.numel() * series_host.element_size() + sum(h.numel() * h.element_size() for h in hosts.values())
    return {"value": val, "unit": UNIT, "h2d_bytes_per_step": cl_host.numel() * cl_host.element_size(),
            "d2h_bytes_per_step": d2h,
            "call": f"twa_run({n_run} KDK steps, moments every {OUT_EVERY}) incl. sampling, then twa_moments of the "
                    "final batch; the scalar series and the final <rho>, <n_k>, Var n_k copied to the host, per step"}


def _max_over_ranks(ms: float, dist, device) -> float:
    """The job's time: the slowest rank's (all_reduce MAX); the local time on one process."""
    if dist is None:
        return ms
    import torch
    t = torch.tensor([ms], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def _tune_cache_path(local_rank: int) -> str:
    """Autotune cache of one GPU of the node (ranks tune concurrently; one file each)."""
    return os.path.join(tempfile.gettempdir(), f"twa_tune_cache_gpu{local_rank}.json")


def run_twa(args):
    import torch
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    from paper_2310_07119_gb300 import Ensemble, twa_advance, twa_last_launch_count, twa_profile_enable, twa_profile_read

    w = _workload(args.streams)
    ns = args.streams
    ens = Ensemble([w.grid], w.phys.hbar_m, w.phys.C, w.phys.dt, w.phys.n_tot, [ns], want_modes=True,
                   device=f"cuda:{local}")
    cl = w.psi_cl()
    tuned = {}
    if not args.no_tune:
        ens.autotune(_tune_cache_path(local))
        try:
            key = f"{GRID_M}x{GRID_M}x{GRID_M}:slots{ns + 1}:"
            tuned = {k[len(key):]: v for k, v in json.load(open(_tune_cache_path(local))).items() if k.startswith(key)}
        except (OSError, ValueError):
            tuned = {}
    ens.sample([cl], w.noise_seed)
    series_w = ens.new_series(max(1, args.warmup) * OUT_EVERY, OUT_EVERY)
    twa_advance(ens.h, ens.psi, max(1, args.warmup) * OUT_EVERY, OUT_EVERY, series_w)
    series = ens.new_series(args.steps * OUT_EVERY, OUT_EVERY)
    st = torch.cuda.current_stream()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)

    def timed(clk_gpu):
        """One timed region of args.steps bench steps (barrier + synchronize on both sides)."""
        torch.cuda.synchronize()
        if dist:
            dist.barrier()
        torch.cuda.synchronize()
        with ClockSampler(clk_gpu) as clk:
            e0.record(st)
            twa_advance(ens.h, ens.psi, args.steps * OUT_EVERY, OUT_EVERY, series)
            e1.record(st)
            torch.cuda.synchronize()
            n_launch = twa_last_launch_count(ens.h)
        if dist:
            dist.barrier()
        torch.cuda.synchronize()
        return _max_over_ranks(e0.elapsed_time(e1), dist, "cuda"), n_launch, clk.summary()

    # headline: the product path, every output interval after the first replayed as a CUDA graph
    ms, launches, clocks = timed(local)
    cell_updates = ns * w.grid.cells * OUT_EVERY * args.steps * world
    value = cell_updates / (ms * 1e-3)
    sc = series.cpu().numpy()
    # the same region again with the pass profiler on (eager launches, each pass bracketed by CUDA
    # events on its stream): per-pass durations for the roofline
    twa_profile_enable(ens.h, True)
    ms_prof, _, clocks_prof = timed(local)
    prof = twa_profile_read(ens.h)
    twa_profile_enable(ens.h, False)

    peak, peak_kind = _peaks()
    dom = max(prof.items(), key=lambda kv: kv[1]["total_ms"])
    name, d = dom
    bytes_per_launch = d["bytes_per_cell"] * d["fields_per_launch"] * d["cells"]
    avg_ms = d["total_ms"] / d["launches"]
    achieved = bytes_per_launch / (avg_ms * 1e-3) / 1e9
    traffic = _ncu_traffic(name)
    passes = {k: {"launches": v["launches"], "avg_ms": v["total_ms"] / v["launches"],
                  "share": v["total_ms"] / sum(x["total_ms"] for x in prof.values()),
                  "GBps": v["bytes_per_cell"] * v["fields_per_launch"] * v["cells"] / (v["total_ms"] / v["launches"] * 1e-3) / 1e9}
              for k, v in prof.items()}
    step_bytes = sum(v["bytes_per_cell"] * v["fields_per_launch"] * v["cells"] * v["launches"] for v in prof.values())
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": f"3D Gaussian-random-field condensation {GRID_M}^3 x {ns} streams (+ classical field), "
                               f"FP32 KDK dt={w.phys.dt:.4e}, moments every {OUT_EVERY} steps",
                   "grid": [GRID_M] * 3, "streams": ns, "kdk_steps_per_step": OUT_EVERY,
                   "batch_bytes": int(ens.psi.numel() * 8), "l2": "inputs larger than L2 (4.2 GB batch)",
                   "path": "twa_advance: graph replay of every output interval after the first",
                   "parallelism": f"replicas x{world}"},
        "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
                     "traffic": traffic, "kernel": name, "peak_kind": f"{peak_kind} copy bandwidth",
                     "bytes_per_launch": bytes_per_launch, "avg_launch_ms": avg_ms},
        "hbm_effective": {"algorithmic_GBps_whole_step": step_bytes / (ms * 1e-3) / 1e9 / world,
                          "frac_of_peak": step_bytes / (ms * 1e-3) / 1e9 / world / peak,
                          "compulsory_16B_frac": 16.0 * cell_updates / world / (ms * 1e-3) / 1e9 / peak,
                          "design_56B_frac": 56.0 * cell_updates / world / (ms * 1e-3) / 1e9 / peak},
        "profiled_eager": {"value": cell_updates / (ms_prof * 1e-3), "unit": UNIT, "ms_per_step": ms_prof / args.steps,
                           "note": "the timed region repeated with the pass profiler on (eager launches, no graph "
                                   "replay); the roofline and per-pass figures come from this run",
                           "clocks": clocks_prof},
        "passes": passes,
        "tuned_passes": {"lines_per_cta_by_axis_op": tuned,
                         "flags": "65536: cp.async-pipelined variant; 131072: two-field variant; axis9 op0: 3D "
                                  "pipeline (0 axis passes, 1 xy-plane passes)"},
        "gpu_launches": int(launches),
        "moments_last": {"Q": float(sc[-1, 0, 0]), "corr": float(sc[-1, 0, 1]), "mass": float(sc[-1, 0, 2])},
        "clocks": clocks,
    }
    if rank == 0 and not args.no_extras and ns == STREAMS:
        line["e2e"] = _e2e(ens, w)
        line["adaptive"] = _adaptive_rate(ens, w)
        line["phase_moments"] = _phase_moments_cost(ens, w)
        line["observable"] = _observable_cost(ens, w)
        line["particles"] = _particles_rate(ens, w)
        ens.close()
        torch.cuda.empty_cache()
        line["f64_plain"] = {"value": _f64_plain_rate(w), "unit": UNIT, "path": "TWA_F64_PLAIN, 1 stream + classical, 128^3"}
        line["cufft_reference"] = {"value": _cufft_reference_rate(w), "unit": UNIT,
                                   "path": "torch.fft (cuFFT) KDK step, 32 fields, reference only"}
        cv, n, el = _oracle_rate(w)
        line["uneven_batch"] = _uneven_rate()
        line["one_d"] = _one_d_rate()
        torch.cuda.empty_cache()
        line["cpu_baseline"] = {"value": cv, "unit": UNIT, "cores": _cores(), "kind": "oracle",
                                "sample": f"2 streams of the 128^3 workload, {n} KDK steps in {el:.1f} s (FP64 scipy.fft)"}
        torch.cuda.empty_cache()
        line["paper_scale_512"] = _paper_scale()
    if rank == 0:
        print(json.dumps(line), flush=True)
    if dist:
        dist.destroy_process_group()


def _ncu_traffic(kernel_op: str):
    """DRAM bytes per launch of the dominant pass from a committed ncu summary, if it was taken on the
    current kernel sources."""
    p = os.path.join(ROOT, "profiles", "ncu_traffic.json")
    if not os.path.exists(p):
        return None
    try:
        d = json.load(open(p))
        from paper_2310_07119_gb300.build import source_digest
        if d.get("source_digest") != source_digest():
            return None
        return d.get("ops", {}).get(kernel_op, {}).get("dram_bytes_per_launch_full_size")
    except Exception:
        return None


def _paper_scale(steps=2, tune=True):
    """512^3 x 64 streams of the stable-object (soliton) workload.  The tuner times every candidate
    pass shape on an 8 GB prefix of the batch (8 of the 65 fields), so tuning takes seconds."""
    import torch
    import twa_inputs as ti
    from paper_2310_07119_gb300 import Ensemble, twa_advance
    w = ti.workload_3d_soliton(512, 64, 4000)
    ens = Ensemble([w.grid], w.phys.hbar_m, w.phys.C, w.phys.dt, w.phys.n_tot, [64], want_modes=True)
    tuned, t_tune = {}, 0.0
    if tune:
        path = _tune_cache_path(torch.cuda.current_device())
        t0 = time.perf_counter()
        ens.autotune(path)
        torch.cuda.synchronize()
        t_tune = time.perf_counter() - t0
        try:
            key = "512x512x512:slots65:"
            tuned = {k[len(key):]: v for k, v in json.load(open(path)).items() if k.startswith(key)}
        except (OSError, ValueError):
            tuned = {}
    ens.sample([w.psi_cl()], w.noise_seed)
    twa_advance(ens.h, ens.psi, OUT_EVERY, OUT_EVERY, ens.new_series(OUT_EVERY, OUT_EVERY))
    series = ens.new_series(steps * OUT_EVERY, OUT_EVERY)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    twa_advance(ens.h, ens.psi, steps * OUT_EVERY, OUT_EVERY, series)
    e1.record()
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1)
    shapes = "tuned pass shapes" if tune else "default pass shapes"
    out = {"workload": f"3D soliton 512^3 x 64 streams (+ classical field), moments every 10 steps, {shapes}",
           "value": 64 * w.grid.cells * OUT_EVERY * steps / (ms * 1e-3), "unit": UNIT, "ms_per_step": ms / steps,
           "batch_bytes": int(ens.psi.numel() * 8), "device_bytes_reserved": int(torch.cuda.memory_reserved())}
    if tune:
        out["tune_seconds"] = round(t_tune, 1)
        out["lines_per_cta_by_axis_op"] = tuned
    ens.close()
    return out


def main():
    args = _args()
    if args.paper_scale:
        print(json.dumps({"paper_scale": _paper_scale()}), flush=True)
        return
    if args.impl == "reference":
        run_reference(args)
    else:
        run_twa(args)


if __name__ == "__main__":
    main()
