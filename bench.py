#!/usr/bin/env python3
"""Throughput benchmark of the pseudo-potential LB step on GB300.

Default workload: D3Q19 BGK, FP32 deviation storage, 256^3 periodic (16.7 M
cells), psi = 1 - exp(-rho), G = -5, 4th-order force stencil, centred droplet
R = 40 (tanh profile rho_l = 2.0, rho_g = 0.15, width 2).  A "step" is one
lattice time step (psi pass + fused stream-collide-force kernel).  Metric:
MLUPS (million lattice updates per second), whole job.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

Under torchrun (N > 1) every rank advances its own replica of the domain (the
single-domain path has no data exchange); the JSON line is printed by rank 0.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

WORKLOADS = {
    # name: lattice, shape (nz, ny, nx), precision, stencil, droplet R
    "d3q19_256_fp32": dict(lattice=1, shape=(256, 256, 256), precision=1, stencil=4, R=40.0,
                           desc="D3Q19 BGK FP32-shifted 256^3 periodic, psi=1-exp(-rho), G=-5, "
                                "4th-order 3-D force stencil, centred droplet R=40"),
    "d3q19_256_fp32_iso6": dict(lattice=1, shape=(256, 256, 256), precision=1, stencil=6, R=40.0,
                                desc="D3Q19 BGK FP32-shifted 256^3 periodic, psi=1-exp(-rho), G=-5, "
                                     "6th-order 3-D force stencil, centred droplet R=40"),
    "d3q19_256_fp32_mrt_iso6": dict(lattice=1, shape=(256, 256, 256), precision=1, stencil=6, R=40.0, collision=1,
                                    desc="D3Q19 MRT (rates 1/tau, s_e=1.64, s_eps=1.54, s_q=1.9) FP32-shifted 256^3 "
                                         "periodic, psi=1-exp(-rho), G=-5, 6th-order 3-D force stencil, centred droplet R=40"),
    "d3q19_256_fp32_mrt": dict(lattice=1, shape=(256, 256, 256), precision=1, stencil=4, R=40.0, collision=1,
                               desc="D3Q19 MRT (rates 1/tau, s_e=1.64, s_eps=1.54, s_q=1.9) FP32-shifted 256^3 "
                                    "periodic, psi=1-exp(-rho), G=-5, 4th-order 3-D force stencil, centred droplet R=40"),
    "d3q19_200_fp32": dict(lattice=1, shape=(200, 200, 200), precision=1, stencil=4, R=31.25,
                           desc="D3Q19 BGK FP32-shifted 200^3 periodic (a row length that is not a power of two), "
                                "psi=1-exp(-rho), G=-5, 4th-order 3-D force stencil, centred droplet R=31.25"),
    "d2q9_8192_fp32_mrt": dict(lattice=0, shape=(1, 8192, 8192), precision=1, stencil=4, R=2048.0, collision=1,
                               desc="D2Q9 MRT (rates 1/tau, s_e=1.64, s_eps=1.54, s_q=1.9) FP32-shifted 8192^2 "
                                    "periodic, psi=1-exp(-rho), G=-5, 4th-order stencil, centred droplet R=2048"),
    "d2q9_8192_fp32": dict(lattice=0, shape=(1, 8192, 8192), precision=1, stencil=4, R=2048.0,
                           desc="D2Q9 BGK FP32-shifted 8192^2 periodic, psi=1-exp(-rho), G=-5, 4th-order stencil, "
                                "centred droplet R=2048"),
    "d2q9_2048_fp64": dict(lattice=0, shape=(1, 2048, 2048), precision=0, stencil=4, R=512.0, alu=True,
                           desc="D2Q9 BGK FP64 2048^2 periodic, psi=1-exp(-rho), G=-5, 4th-order stencil, "
                                "centred droplet R=512 (FP64-ALU-bound on GB300)"),
    "d2q9_64_fp64": dict(lattice=0, shape=(1, 64, 64), precision=0, stencil=4, R=16.0,
                         desc="D2Q9 BGK FP64 64^2 periodic, psi=1-exp(-rho), G=-5, 4th-order stencil, "
                              "centred droplet R=16"),
}
RHO_L, RHO_G, WIDTH, G, TAU = 2.0, 0.15, 2.0, -5.0, 1.0
HBM_FALLBACK_GBS = 6800.0
# No FP64 peak is measured on this machine; the nominal GB300 FP64 rate (non-tensor)
# is the ALU roofline of the FP64 step.
FP64_NOMINAL_GFLOPS = 1250.0


def measured_peak_gbs():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as fh:
            return float(json.load(fh)["hbm_gbs"]), "measured"
    except Exception:
        return HBM_FALLBACK_GBS, "fallback"


def kernel_source_hash():
    """Hash of the sources that define the single-domain step kernels (the ones
    the recorded counters describe); the batch, network and API files are not
    part of it."""
    h = hashlib.sha256()
    csrc = os.path.join(ROOT, "paper_1906_11027_gb300", "csrc")
    for fn in sorted(os.listdir(csrc)):
        if fn in ("kernels.cuh", "lattice.cuh", "internal.h") or (fn.startswith("kernels_") and fn.endswith(".cu")):
            with open(os.path.join(csrc, fn), "rb") as fh:
                h.update(fn.encode())
                h.update(fh.read())
    return h.hexdigest()[:16]


def recorded_traffic(kernel, workload):
    """DRAM bytes per launch from the committed ncu summary, if it was taken on
    the current kernel sources; else None."""
    path = os.path.join(ROOT, "profiles", "dram_traffic.json")
    try:
        with open(path) as fh:
            rec = json.load(fh)
        e = rec[workload][kernel]
        if e.get("source_hash") != kernel_source_hash():
            return None
        return float(e["bytes_per_launch"])
    except Exception:
        return None


def recorded_flops(kernel, workload):
    """FP64 flops per cell from the committed ncu instruction counts, if they were
    taken on the current kernel sources; else None."""
    path = os.path.join(ROOT, "profiles", "fp64_flops.json")
    try:
        with open(path) as fh:
            e = json.load(fh)[workload][kernel]
        if e.get("source_hash") != kernel_source_hash():
            return None
        return float(e["flops_per_cell"])
    except Exception:
        return None


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device_index):
        self.device_index = device_index
        self.proc = None
        self.lines = []
        self._t = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.device_index}", f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "100"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None
            return
        self._t = threading.Thread(target=self._read, daemon=True)
        self._t.start()

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"], "samples": 0}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        if self._t:
            self._t.join(timeout=2)
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        return {"sm_mhz": float(np.median(sm)) if sm else None,
                "sm_max_mhz": float(max(smax)) if smax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


def dist_setup(args):
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch
        import torch.distributed as dist
        torch.cuda.set_device(local)
        backend = "nccl" if args.impl == "ours" else "gloo"
        dist.init_process_group(backend=backend)
    return world, rank, local


def barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def max_over_ranks(x, world):
    """Largest value over the ranks (the slowest rank's time)."""
    if world == 1:
        return x
    import torch
    import torch.distributed as dist
    dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
    t = torch.tensor([x], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_mlups(world, cells_per_rank, steps, max_elapsed_ms):
    """Whole-job throughput of `world` replicas, timed by the slowest rank."""
    return world * cells_per_rank * steps / (max_elapsed_ms * 1e-3) / 1e6


def oracle_sample_run(wl, budget_s, steps, fill_budget=False):
    """Time the FP64 oracle for `steps` steps on a box of the workload's lattice,
    stencil and droplet, its side chosen so the run takes about budget_s (capped
    at the workload's own side; with fill_budget the step count then grows to
    fill the budget).

    Returns (MLUPS, sample description, cores, seconds)."""
    import oracle
    nz, ny, nx = wl["shape"]
    dim = 3 if nz > 1 else 2
    lat = {0: oracle.D2Q9, 1: oracle.D3Q19}[wl["lattice"]]
    side = 48 if dim == 3 else 64
    coll = {0: oracle.BGK, 1: oracle.MRT}[wl.get("collision", 0)]
    probe = oracle.Sim(lat, side, side, side if dim == 3 else 1, stencil=wl["stencil"], G=G, tau=TAU, coll=coll)
    probe.init_droplet(RHO_L, RHO_G, wl["R"] * side / nx, WIDTH)
    t0 = time.perf_counter()
    probe.step(2)
    rate = 2 * probe.N / (time.perf_counter() - t0)  # cell updates per second
    del probe
    L = int((budget_s * rate / steps) ** (1.0 / dim))
    L = max(16, min(nx, (L // 8) * 8))
    if fill_budget:
        steps = max(steps, int(budget_s * rate / L ** dim))
    sim = oracle.Sim(lat, L, L, L if dim == 3 else 1, stencil=wl["stencil"], G=G, tau=TAU, coll=coll)
    sim.init_droplet(RHO_L, RHO_G, wl["R"] * L / nx, WIDTH)
    t0 = time.perf_counter()
    sim.step(steps)
    dt = time.perf_counter() - t0
    mlups = sim.N * steps / dt / 1e6
    cores = int(os.environ.get("OMP_NUM_THREADS", os.cpu_count() or 1))
    sample = (f"FP64 oracle on a {L}^{dim} box of the same lattice, stencil and droplet "
              f"(R scaled by {L}/{nx}), {steps} steps in {dt:.1f} s")
    return mlups, sample, cores, dt


def oracle_single_thread(workload, budget_s):
    """The same oracle sample on one host thread, in a child process (OpenMP
    reads its thread count when the library starts)."""
    env = dict(os.environ, OMP_NUM_THREADS="1")
    try:
        out = subprocess.run([sys.executable, os.path.abspath(__file__), "--oracle-sample", workload,
                              "--cpu-budget", str(budget_s)], env=env, capture_output=True, text=True,
                             timeout=20 * budget_s + 120)
        return json.loads([l for l in out.stdout.splitlines() if l.startswith("{")][-1])
    except Exception as e:  # report the failure instead of a number
        return {"error": str(e)[:200]}


def run_reference(args, world, rank):
    """The oracle arm: the FP64 CPU oracle, as it stands, on the host cores."""
    if rank != 0:
        return 0
    wl = WORKLOADS[args.workload]
    nsteps = args.steps + args.warmup
    mlups, sample, cores, dt = oracle_sample_run(wl, 120.0, nsteps)
    line = {
        "impl": "reference", "metric": "MLUPS", "value": round(mlups, 4), "unit": "MLUPS",
        "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": round(1e3 * dt / nsteps, 4), "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": args.workload, "desc": wl["desc"]},
        "cpu_baseline": {"value": round(mlups, 4), "unit": "MLUPS", "cores": cores, "kind": "oracle",
                         "sample": sample},
        "e2e": {"value": round(mlups, 4), "unit": "MLUPS", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


def run_ours(args, world, rank, local):
    import torch
    from paper_1906_11027_gb300 import lbm

    torch.cuda.set_device(local)
    lbm.load()
    wl = WORKLOADS[args.workload]
    nz, ny, nx = wl["shape"]
    cells = nx * ny * nz
    stream = torch.cuda.Stream()
    path = {"auto": lbm.LBM_PATH_AUTO, "two": lbm.LBM_PATH_TWO_PASS, "one": lbm.LBM_PATH_ONE_PASS}[args.path]
    dom = lbm.Domain(nx, ny, nz, lattice=wl["lattice"], stencil=wl["stencil"], G=G, tau=TAU,
                     collision=wl.get("collision", lbm.LBM_BGK),
                     precision=wl["precision"], stream=stream, torch_alloc=True, path=path)
    if args.schedule:  # pin a schedule (profiling runs), else the autotuner picks
        dom.set_schedule(args.schedule)
    dom.init_droplet(RHO_L, RHO_G, wl["R"], WIDTH)
    dom.step(args.warmup)
    torch.cuda.synchronize()
    barrier(world)

    sampler = ClockSampler(local)
    sampler.start()
    time.sleep(0.3)  # let the sampler attach before the timed region
    ev0 = torch.cuda.Event(enable_timing=True)
    ev1 = torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    ev0.record(stream)
    kernel_ms = dom.step_timed(args.steps)  # CUDA events around every kernel, same stream
    ev1.record(stream)
    torch.cuda.synchronize()
    clocks = sampler.stop()
    elapsed_ms = ev0.elapsed_time(ev1)
    schedule = dom.schedule_report()
    barrier(world)
    elapsed_ms = max_over_ranks(elapsed_ms, world)
    ms_per_step = elapsed_ms / args.steps
    value = job_mlups(world, cells, args.steps, elapsed_ms)

    # roofline of the dominant kernel
    peak, peak_src = measured_peak_gbs()
    s = 4 if wl["precision"] == 1 else 8
    Q = lbm.Q_OF[wl["lattice"]]
    kept = 1 if s == 8 else 0  # the FP64 step keeps the density between its kernels
    per_cell = {"k_fused": (2 * Q + 1 + kept) * s, "k_psi": (Q + 1 + kept) * s, "k_onepass": 2 * Q * s}
    dom_k = max(kernel_ms, key=kernel_ms.get)
    b_alg = dom.bytes_per_update()
    # the dominant kernel against the step's algorithmic bytes per update,
    # B_alg = 2 Q s + 2 s (one read and write of every population, one write
    # and read of psi); when one kernel is the whole step (the one-pass
    # schedules) this is the step's roofline, met without the psi traffic
    alg_cell = b_alg if len(kernel_ms) == 1 else per_cell[dom_k]
    achieved = alg_cell * cells / (kernel_ms[dom_k] * 1e-3) / 1e9
    achieved_own = per_cell[dom_k] * cells / (kernel_ms[dom_k] * 1e-3) / 1e9
    traffic = recorded_traffic(dom_k, args.workload)
    step_gbs = value / world * 1e6 * b_alg / 1e9

    # end to end through the public API with host buffers: upload the initial
    # density from pinned host memory, step, read the observables back
    rho_host = torch.empty(cells, dtype=torch.float64, pin_memory=True).numpy()
    z, y, x = np.meshgrid(np.arange(nz) - nz // 2, np.arange(ny) - ny // 2, np.arange(nx) - nx // 2,
                          indexing="ij")
    r = np.sqrt(x * x + y * y + (z * z if nz > 1 else 0)).ravel()
    rho_host[:] = 0.5 * (RHO_L + RHO_G) - 0.5 * (RHO_L - RHO_G) * np.tanh(2 * (r - wl["R"]) / WIDTH)
    del x, y, z, r
    e2e_steps = args.steps
    torch.cuda.synchronize()
    barrier(world)
    t0 = time.perf_counter()
    dom.init_from_rho(rho_host)
    dom.step(e2e_steps)
    obs = dom.observables()
    e2e_s = time.perf_counter() - t0
    e2e_s = max_over_ranks(e2e_s, world)
    e2e_value = world * cells * e2e_steps / e2e_s / 1e6
    d2h = (16 + nx) * 8 + 4

    line = {
        "metric": "MLUPS", "value": round(value, 2), "unit": "MLUPS", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(ms_per_step, 5),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f32" if wl["precision"] == 1 else "f64", "data": "synthetic",
        "config": {"workload": args.workload, "desc": wl["desc"], "cells": cells,
                   "parallelism": f"replicas{world}" if world > 1 else "single",
                   "l2": "inputs larger than L2 (populations %.2f GB)" % (2 * Q * s * cells / 1e9),
                   "schedule": schedule},
        "roofline": {"bound": "hbm", "kernel": dom_k, "achieved": round(achieved, 1), "peak": peak,
                     "unit": "GB/s", "frac": round(achieved / peak, 4), "traffic": traffic,
                     "algorithmic_bytes_per_cell": alg_cell, "peak_source": peak_src,
                     "kernel_own_bytes_per_cell": per_cell[dom_k],
                     "frac_of_kernel_own_bytes": round(achieved_own / peak, 4),
                     "kernel_ms": {k: round(v, 5) for k, v in kernel_ms.items()}},
        "step_roofline": {"bytes_per_update": b_alg, "achieved_gbs": round(step_gbs, 1),
                          "frac": round(step_gbs / peak, 4),
                          "roofline_mlups": round(peak * 1e9 / b_alg / 1e6, 1)},
        "clocks": clocks,
        "gpu_launches": len(kernel_ms) * args.steps,
        "e2e": {"value": round(e2e_value, 2), "unit": "MLUPS",
                "h2d_bytes_per_step": round(8 * cells / e2e_steps, 1),
                "d2h_bytes_per_step": round(d2h / e2e_steps, 1),
                "note": f"init_from_rho(host) + step({e2e_steps}) + observables(); mass {obs['mass']:.6e}"},
    }
    dom.close()
    if wl.get("alu"):
        # FP64 on GB300: the step is bound by FP64 arithmetic, not by HBM
        fpc = recorded_flops(dom_k, args.workload)
        gflops = fpc * cells / (kernel_ms[dom_k] * 1e-3) / 1e9 if fpc else None
        line["roofline"] = {
            "bound": "alu", "kernel": dom_k, "achieved": round(gflops, 1) if gflops else None,
            "peak": FP64_NOMINAL_GFLOPS, "unit": "GFLOP/s",
            "frac": round(gflops / FP64_NOMINAL_GFLOPS, 4) if gflops else None, "traffic": traffic,
            "flops_per_cell": fpc, "peak_source": "nominal GB300 FP64 rate (no measured FP64 peak)",
            "hbm_context": {"achieved_gbs": round(achieved, 1), "frac_of_measured_copy": round(achieved / peak, 4)},
            "kernel_ms": {k: round(v, 5) for k, v in kernel_ms.items()}}
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        mlups, sample, cores, _ = oracle_sample_run(wl, args.cpu_budget, 4, fill_budget=True)
        line["cpu_baseline"] = {"value": round(mlups, 3), "unit": "MLUPS", "cores": cores, "kind": "oracle",
                                "sample": sample,
                                "single_thread": oracle_single_thread(args.workload, args.cpu_budget / 2)}
    if rank == 0 and world == 1 and not args.no_sweep:
        line["sweep"] = sweep_summary(args)
    if rank == 0:
        print(json.dumps(line), flush=True)
    return 0


def sweep_compare(args, n_domains, with_warm, train_domains, epochs, details):
    """Batched FP32 sweep (one persistent-kernel CUDA graph for all domains) against
    plain FP64 one-domain-per-launch runs of the same domains, both to steady state
    (paper_1906_11027_gb300.sweep).  With with_warm the batched sweep also runs
    from the learned warm start, the network trained beforehand on the steady
    states of a separate draw of domains (another seed), so the timed domains are
    unseen.  Every domain's steady max|u| is classified by the sweep's agreement
    rule.  Returns the result line (a dict)."""
    import torch
    from paper_1906_11027_gb300 import inputs, lbm, sweep, warmstart

    lbm.load()
    doms = inputs.sweep_domains(n_domains)
    cells = sum(d["nx"] * d["ny"] for d in doms)
    torch.cuda.synchronize()
    # warm the kernels (module load) outside the timed regions
    w = lbm.Batch(doms[:2], precision=lbm.LBM_FP32_SHIFTED)
    w.step(4)
    w.close()
    net, train_info = None, None
    if with_warm:
        t0 = time.perf_counter()
        tdoms = inputs.sweep_domains(train_domains, seed=inputs.SWEEP_SEED + 1)
        tb = lbm.Batch(tdoms, precision=lbm.LBM_FP32_SHIFTED)
        _, tobs, _ = tb.run_to_steady(sweep.TOL, args.sweep_max_steps, sweep.K)
        Xt, yt, Xv, yv, _ = warmstart.dataset_from_batch(tb, tdoms, tobs)
        tb.close()
        t_gen = time.perf_counter() - t0
        t0 = time.perf_counter()
        net, loss = warmstart.train(Xt, yt, epochs=epochs)
        torch.cuda.synchronize()
        train_info = {"train_domains": len(tdoms), "train_seed": inputs.SWEEP_SEED + 1,
                      "train_samples": int(len(yt)), "profile_sweep_s": round(t_gen, 2),
                      "train_s": round(time.perf_counter() - t0, 2), "train_loss": loss,
                      "val_mse": float(np.mean((net.predict(Xv) - yv) ** 2)) if len(yv) else None}

    plain = sweep.batched(doms, None, args.sweep_max_steps, args.fp64_below)
    warm = sweep.batched(doms, net, args.sweep_max_steps, args.fp64_below) if with_warm else None
    ref = sweep.one_per_launch(doms, args.sweep_max_steps, sweep.misses_5pct(*[a for a in (plain, warm) if a]))
    cls_t = sweep.classify(doms, plain, ref, args.fp64_below)
    cls_w = sweep.classify(doms, warm, ref, args.fp64_below, tanh_arm=plain) if warm else None
    for arm in (plain, warm):
        if arm:
            arm["batch"].close()
    main_arm = warm if warm else plain
    cls = cls_w if warm else cls_t
    obs32, obs64, steps32, steps64 = main_arm["obs"], ref["obs"], main_arm["steps"], ref["steps"]
    finite = [i for i in range(len(doms)) if np.isfinite(obs64[i]["max_u"]) and np.isfinite(obs32[i]["max_u"])]
    ratio = [abs(obs32[i]["max_u"] / obs64[i]["max_u"] - 1.0) for i in finite] or [float("nan")]
    arms = {"batched_fp32_tanh_s": round(plain["t"], 3),
            "tanh_fp32_phase_s": round(plain["t_fp32"], 3),
            "diverged_tanh_fp32": sum(1 for o in plain["obs"] if not np.isfinite(o["max_u"])),
            "steps_total_tanh": int(sum(plain["steps"]))}
    if warm:
        both = [i for i in range(len(doms)) if np.isfinite(plain["obs"][i]["max_u"])
                and np.isfinite(warm["obs"][i]["max_u"]) and plain["steps"][i] < args.sweep_max_steps
                and warm["steps"][i] < args.sweep_max_steps]
        arms.update({"batched_fp32_warm_s": round(warm["t"], 3), "warm_init_s": round(warm["t_init"], 3),
                     "warm_fp32_phase_s": round(warm["t_fp32"], 3),
                     "warm_fallbacks": warm["fallbacks"], "warm_restarted_from_tanh": warm["restarted"],
                     "steps_total_warm": int(sum(warm["steps"])),
                     "converged_in_both": len(both),
                     "steps_converged_in_both": {"tanh": int(sum(plain["steps"][i] for i in both)),
                                                 "warm": int(sum(warm["steps"][i] for i in both))}})
    line = {
        "metric": "sweep_time_to_steady_s", "value": round(main_arm["t"], 3), "unit": "s", "higher_is_better": False,
        "n_gpus": 1, "dtype": "f32", "data": "synthetic",
        "config": {"workload": "d2q9_sweep_warm" if warm else "d2q9_sweep", "domains": len(doms), "cells": cells,
                   "seed": inputs.SWEEP_SEED, "batch_tile": main_arm["schedule"],
                   "rule": "|max|u|(t) - max|u|(t-100)| / 100 < 1e-10 (FP32 adds the floor 1e-6 max|u|/100), "
                           "checked every 100 steps in both arms",
                   "fp64_below": args.fp64_below, "promoted_to_fp64": main_arm["tiny"],
                   "max_steps": args.sweep_max_steps},
        "baseline_fp64_one_domain_per_launch_s": round(ref["t"], 3),
        "speedup": round(ref["t"] / main_arm["t"], 2),
        "converged": {"batched_fp32": bool(main_arm["ok"]),
                      "fp64": sum(1 for s in steps64 if s < args.sweep_max_steps)},
        "steps": {"batched_fp32_total": int(sum(steps32)), "fp64_total": int(sum(steps64))},
        "diverged": {"fp64": sum(1 for o in obs64 if not np.isfinite(o["max_u"])),
                     "batched_fp32": sum(1 for o in obs32 if not np.isfinite(o["max_u"]))},
        "per_domain_columns": ["L", "G", "tau", "order", "R", "steps_batched", "steps_fp64", "max_u_batched",
                               "max_u_fp64", "steps_tanh_fp32", "max_u_tanh_fp32", "class", "class_tanh"],
        "per_domain": [[d["nx"], round(d["G"], 3), d["tau"], d["stencil"], round(d["R"], 1), int(steps32[i]),
                        int(steps64[i]), float("%.4g" % obs32[i]["max_u"]), float("%.4g" % obs64[i]["max_u"]),
                        int(plain["steps"][i]), float("%.4g" % plain["obs"][i]["max_u"]), cls[i], cls_t[i]]
                       for i, d in enumerate(doms)] if details else None,
        "max_u_rel_diff": {"max": round(max(ratio), 4), "median": round(float(np.median(ratio)), 4),
                           "compared": len(finite), "classes": sweep.counts(cls)},
        "max_u_rel_diff_tanh_fp32_vs_fp64": {"classes": sweep.counts(cls_t)},
        "arms": arms,
        "warm_start_training": train_info,
    }
    return line


def run_sweep(args):
    line = sweep_compare(args, args.sweep_domains, args.sweep_warm, args.ws_train_domains, args.ws_epochs,
                         args.sweep_details)
    print(json.dumps(line), flush=True)
    return 0


def sweep_summary(args):
    """The sweep half of the metric, bounded for the default line: a
    --sweep-sub-domains draw of the parameter sweep (seed 11027), batched FP32
    from the tanh and from the learned start (network trained first on an
    equal draw of seed 11028) against plain FP64 one domain per launch, all to
    steady state, with the per-domain max|u| agreement classified."""
    t0 = time.perf_counter()
    ln = sweep_compare(args, args.sweep_sub_domains, True, args.sweep_sub_domains, args.sweep_sub_epochs, False)
    a = ln["arms"]
    return {
        "metric": "sweep_time_to_steady_s", "unit": "s", "domains": ln["config"]["domains"],
        "cells": ln["config"]["cells"], "seed": ln["config"]["seed"],
        "batched_fp32_tanh_s": a["batched_fp32_tanh_s"], "batched_fp32_warm_s": a["batched_fp32_warm_s"],
        "warm_init_s": a["warm_init_s"], "fp64_one_domain_per_launch_s": ln["baseline_fp64_one_domain_per_launch_s"],
        "speedup_tanh": round(ln["baseline_fp64_one_domain_per_launch_s"] / a["batched_fp32_tanh_s"], 2),
        "speedup_warm": ln["speedup"],
        "steps_total": {"tanh_fp32": a["steps_total_tanh"], "warm_fp32": a["steps_total_warm"],
                        "fp64": ln["steps"]["fp64_total"]},
        "steps_converged_in_both": a["steps_converged_in_both"],
        "warm_restarted_from_tanh": a["warm_restarted_from_tanh"],
        "agreement_classes_warm_vs_fp64": ln["max_u_rel_diff"]["classes"],
        "agreement_classes_tanh_vs_fp64": ln["max_u_rel_diff_tanh_fp32_vs_fp64"]["classes"],
        "warm_start_training": ln["warm_start_training"],
        "rule": ln["config"]["rule"],
        "wall_s": round(time.perf_counter() - t0, 1),
    }


def run_warmstart(args):
    """Learned warm start: batched sweep -> steady profiles -> network trained on the
    GPU (held-out domains for validation) -> plain tanh vs learned start on
    held-out domains, a D2Q9 512^2 droplet and a D3Q19 128^3 droplet."""
    import torch
    from paper_1906_11027_gb300 import inputs, lbm, warmstart

    lbm.load()
    doms = inputs.sweep_domains(args.ws_sweep_domains)
    t0 = time.perf_counter()
    b = lbm.Batch(doms, precision=lbm.LBM_FP32_SHIFTED)
    steps, obs, _ = b.run_to_steady(1e-10, args.sweep_max_steps, 100)
    t_sweep = time.perf_counter() - t0
    Xt, yt, Xv, yv, held = warmstart.dataset_from_batch(b, doms, obs)
    b.close()
    t0 = time.perf_counter()
    net, loss = warmstart.train(Xt, yt, epochs=args.ws_epochs)
    torch.cuda.synchronize()
    t_train = time.perf_counter() - t0
    val_mse = float(np.mean((net.predict(Xv) - yv) ** 2)) if len(yv) else None

    def compare(make, init_plain, init_warm, tol, max_steps):
        out = {}
        for mode in ("plain", "warm"):
            dom = make()
            t1 = time.perf_counter()
            fb = None
            if mode == "plain":
                init_plain(dom)
            else:
                fb, _ = init_warm(dom)
            s, ok = dom.run_to_steady(tol, max_steps, 100)
            torch.cuda.synchronize()
            dt = time.perf_counter() - t1
            o = dom.observables()
            out[mode] = dict(steps=s, ok=ok, s=dt, max_u=o["max_u"], rho=dom.fields()["rho"], fallback=fb)
            dom.close()
        return {"steps_plain": out["plain"]["steps"], "steps_warm": out["warm"]["steps"],
                "time_plain_s": round(out["plain"]["s"], 3), "time_warm_s": round(out["warm"]["s"], 3),
                "converged": [out["plain"]["ok"], out["warm"]["ok"]], "fallback": out["warm"]["fallback"],
                "max_abs_drho": float(np.abs(out["plain"]["rho"] - out["warm"]["rho"]).max()),
                "max_u_rel_diff": abs(out["warm"]["max_u"] / out["plain"]["max_u"] - 1.0)}

    heldout = []
    for i in held[:args.ws_heldout]:
        d = doms[i]
        r = compare(lambda d=d: lbm.Domain(d["nx"], d["ny"], G=d["G"], tau=d["tau"], stencil=d["stencil"]),
                    lambda dom, d=d: dom.init_droplet(d["rho_l"], d["rho_g"], d["R"], d["width"]),
                    lambda dom, d=d: dom.init_droplet_learned(net, d["R"], d["rho_l"], d["rho_g"], d["width"]),
                    1e-13, 600000)
        r.update(L=d["nx"], G=round(d["G"], 3), tau=d["tau"], order=d["stencil"], R=round(d["R"], 1))
        heldout.append(r)
    big2 = compare(lambda: lbm.Domain(512, 512, G=-5.0, tau=1.0, stencil=4),
                   lambda dom: dom.init_droplet(2.0, 0.15, 100.0, 2.0),
                   lambda dom: dom.init_droplet_learned(net, 100.0, 2.0, 0.15, 2.0), 1e-13, 900000)
    # FP64 in 3-D too: the 1e-6 density match needs the slow relaxation resolved
    # below FP32's round-off floor
    big3 = compare(lambda: lbm.Domain(128, 128, 128, lattice=lbm.LBM_D3Q19, G=-5.0, tau=1.0,
                                      precision=lbm.LBM_FP64),
                   lambda dom: dom.init_droplet(2.0, 0.15, 30.0, 2.0),
                   lambda dom: dom.init_droplet_learned(net, 30.0, 2.0, 0.15, 2.0), 1e-13, 400000)
    used = [h for h in heldout if not h["fallback"]]
    line = {
        "metric": "warm_start_steps_saved", "unit": "fraction of plain steps",
        "value": round(float(np.mean([1 - h["steps_warm"] / h["steps_plain"] for h in used])), 4) if used else None,
        "higher_is_better": True, "n_gpus": 1, "dtype": "bf16/f32 network, f64 runs", "data": "synthetic",
        "config": {"workload": "learned_warm_start", "sweep_domains": len(doms), "train_samples": int(len(yt)),
                   "val_samples": int(len(yv)), "heldout_domains": len(held), "epochs": args.ws_epochs},
        "sweep_s": round(t_sweep, 2), "train_s": round(t_train, 2), "train_loss": loss, "val_mse": val_mse,
        "steady_rule": "|max|u|(t) - max|u|(t-100)| / 100 < 1e-13, FP64 runs",
        "heldout": heldout, "d2q9_512": big2, "d3q19_128_fp64": big3,
    }
    print(json.dumps(line), flush=True)
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3000)
    ap.add_argument("--warmup", type=int, default=20)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--workload", choices=sorted(WORKLOADS), default="d3q19_256_fp32")
    ap.add_argument("--cpu-budget", type=float, default=15.0)
    ap.add_argument("--path", choices=["auto", "two", "one"], default="auto")
    ap.add_argument("--schedule", default=None, help="pin the step schedule by name instead of autotuning")
    ap.add_argument("--sweep", action="store_true", help="time the batched sweep instead of the step")
    ap.add_argument("--sweep-domains", type=int, default=64)
    ap.add_argument("--no-sweep", action="store_true",
                    help="leave the bounded sweep comparison out of the step benchmark's line")
    ap.add_argument("--sweep-sub-domains", type=int, default=64,
                    help="domains of the sweep comparison carried by the step benchmark's line")
    ap.add_argument("--sweep-sub-epochs", type=int, default=40)
    ap.add_argument("--sweep-max-steps", type=int, default=200000)
    ap.add_argument("--sweep-details", action="store_true")
    ap.add_argument("--sweep-warm", action="store_true",
                    help="batched arm starts from the learned warm start (network trained first on another draw)")
    ap.add_argument("--ws-train-domains", type=int, default=256,
                    help="domains of the separate draw the sweep's warm-start network is trained on")
    ap.add_argument("--ws-sweep-domains", type=int, default=256,
                    help="sweep domains whose steady states train the network of --warmstart")
    ap.add_argument("--warmstart", action="store_true", help="train and evaluate the learned warm start")
    ap.add_argument("--ws-epochs", type=int, default=80)
    ap.add_argument("--ws-heldout", type=int, default=12)
    ap.add_argument("--fp64-below", type=float, default=1e-6,
                    help="steady max|u| under which an FP32 domain is re-converged in FP64")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--oracle-sample", default=None, help=argparse.SUPPRESS)
    args = ap.parse_args()
    if args.oracle_sample:  # child of oracle_single_thread: one sample, one JSON line
        mlups, sample, cores, dt = oracle_sample_run(WORKLOADS[args.oracle_sample], args.cpu_budget, 2,
                                                     fill_budget=True)
        print(json.dumps({"value": round(mlups, 3), "unit": "MLUPS", "cores": cores, "sample": sample}))
        return 0
    if args.warmup < 3:
        ap.error("--warmup must be >= 3")
    if args.sweep:
        return run_sweep(args)
    if args.warmstart:
        return run_warmstart(args)
    world, rank, local = dist_setup(args)
    try:
        if args.impl == "reference":
            return run_reference(args, world, rank)
        return run_ours(args, world, rank, local)
    finally:
        if world > 1:
            import torch.distributed as dist
            dist.destroy_process_group()


if __name__ == "__main__":
    sys.exit(main())
