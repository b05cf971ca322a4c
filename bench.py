#!/usr/bin/env python3
"""Benchmark of the two-component D2Q9 Shan-Chen LB time step on GB300.

Workload (N = 1): 1024 x 2048 grid, FP32 populations, tau 1, G 1.4 (immiscible),
masses 1.0 / 0.9, g 1e-5, 8-mode interface; one benchmark step = 100 LB time
steps plus one diagnostics evaluation (energy-budget terms every 100 steps).
The metric is MLUPS (million lattice-site updates per second; one update
advances both components).  Population buffers (2 x 151 MB) exceed the 129 MB
L2, so no separate L2 flush is needed between steps.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
                  [--storage f32|f16|bf16]
                  [--kernel staged|paired|decoupled|warp|pipe|fused|two_pass]
                  [--tile-y T] [--nx NX --ny NY] [--ensemble M] [--storage-study STEPS]
                  [--paper-case STEPS] [--closure-accuracy] [--closure] [--no-extra-lines]

--impl reference times the FP64 CPU oracle on the host on a bounded sample of
the same workload.  With torchrun (N > 1) every rank advances its own
independent realisation (replicas, no collective on the data path); the time is
the maximum over ranks and the value is the whole-job rate.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import time
from pathlib import Path

ROOT = Path(__file__).resolve().parent
sys.path.insert(0, str(ROOT))

LB_STEPS_PER_STEP = 100
BYTES_PER_SITE = {"f32": 144, "f16": 72, "bf16": 72}   # 18 loads + 18 stores per site update
METRIC = "MLUPS & HBM-roofline %; plain FP32 vs FP16-store/ensemble/learned @ stated err"
PROFILE_TRAFFIC = ROOT / "profiles" / "traffic.json"


def workload(args) -> dict:
    return dict(nx=args.nx, ny=args.ny, tau_A=1.0, tau_B=1.0, G=1.4, mass_A=1.0, mass_B=0.9, g=1e-5,
                n_modes=8, amp=2.0, width=1.5, minority=0.08, crop_rows=10)


def l2_note(buffer_bytes: int) -> str:
    """How the timed steps relate to the 129 MB L2: each LB step reads one population
    buffer and writes the other, so the two together are what could stay cached."""
    both = 2 * buffer_bytes
    size = f"two population buffers of {buffer_bytes / 1e6:.0f} MB each, {both / 1e6:.0f} MB together, vs 129 MB L2"
    if both > 129e6:
        return f"inputs larger than L2 ({size}; each LB step reads one buffer and writes the other)"
    return f"inputs fit in L2 ({size}): no L2 flush between steps, so this is not a DRAM-bound figure"


def config_of(args, n_gpus) -> dict:
    return {
        "workload": f"{args.nx}x{args.ny} two-component D2Q9 Shan-Chen Rayleigh-Taylor, G=1.4, tau=1, "
                    f"{args.storage} populations, diagnostics every {LB_STEPS_PER_STEP} steps",
        "nx": args.nx, "ny": args.ny, "lb_steps_per_step": LB_STEPS_PER_STEP,
        "storage": args.storage, "kernel": args.kernel, "tile_y": args.tile_y,
        "l2": l2_note(args.nx * args.ny * BYTES_PER_SITE[args.storage] // 2),
        "parallelism": f"replicas{n_gpus}" if n_gpus > 1 else "single",
    }


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


STEP_SOURCES = ("step_kernels.cu", "collide.cuh", "lattice.cuh", "lbm_internal.cuh")


def kernel_source_hash() -> str:
    """Hash of the sources the step kernels are compiled from."""
    h = hashlib.sha256()
    for name in STEP_SOURCES:
        h.update((ROOT / "paper_2101_04847_gb300" / "csrc" / name).read_bytes())
    return h.hexdigest()[:16]


def profiled_traffic(kernel_name: str, nx: int, ny: int):
    """DRAM bytes per launch of the dominant kernel from the committed ncu summary, scaled
    to this grid; None when absent or taken on a different kernel source."""
    try:
        d = json.loads(PROFILE_TRAFFIC.read_text())
    except (OSError, ValueError):
        return None
    e = d.get(kernel_name)
    if not e or e.get("source_hash") != kernel_source_hash():
        return None
    return e["dram_bytes_per_launch"] * (nx * ny) / (e["nx"] * e["ny"])


class ClockSampler:
    """nvidia-smi clocks / throttle reasons sampled every 200 ms during the timed region."""

    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.path = Path(os.environ.get("TMPDIR", "/tmp")) / f"bench_clocks_{os.getpid()}.csv"

    def __enter__(self):
        try:
            self.out = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.QUERY}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=self.out, stderr=subprocess.DEVNULL)
        except OSError:
            self.proc = None
        return self

    def __exit__(self, *exc):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
            self.out.close()

    def summary(self):
        if self.proc is None:
            return None
        rows = []
        for line in self.path.read_text().splitlines():
            parts = [x.strip() for x in line.split(",")]
            if len(parts) >= 9:
                rows.append(parts)
        try:
            self.path.unlink()
        except OSError:
            pass
        if not rows:
            return None
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({n for r in rows for n, v in zip(names, r[5:9]) if v.lower() == "active"})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(rows)}


def replica_seed(rank: int) -> int:
    """Each rank advances its own independent realisation (the paper's ensembles are
    independent runs), seeded 1, 2, ... by rank."""
    return 1 + rank


def max_over_ranks(values, device=None):
    """Element-wise maximum of a list of floats over all ranks (identity on one rank)."""
    import torch
    import torch.distributed as dist

    if not dist.is_available() or not dist.is_initialized() or dist.get_world_size() == 1:
        return list(values)
    t = torch.tensor(list(values), dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return t.tolist()


def measured_peak_hbm():
    try:
        d = json.loads((ROOT / "MEASURED_PEAKS.json").read_text())
        return float(d["hbm_gbs"]), "measured"
    except (OSError, ValueError, KeyError):
        return 6800.0, "fallback"


# ---------------------------------------------------------------------------
def run_ours(args):
    import torch
    import torch.distributed as dist

    from paper_2101_04847_gb300 import lbm

    ws, rank, local = dist_env()
    torch.cuda.set_device(local)
    if ws > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    params = workload(args)
    params["seed"] = replica_seed(rank)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        solver = lbm.Solver(storage=args.storage, kernel=args.kernel, tile_y=args.tile_y, **params)
    sites = args.nx * args.ny
    launches_per_step = LB_STEPS_PER_STEP * (2 if args.kernel == "two_pass" else 1) + 2   # the diagnostics: a sweep and a reduction

    def one_step(ev_pair=None):
        if ev_pair is not None:
            ev_pair[0].record(stream)
        solver.step(LB_STEPS_PER_STEP)
        if ev_pair is not None:
            ev_pair[1].record(stream)
        solver.diagnostics()

    for _ in range(args.warmup):
        one_step()
    torch.cuda.synchronize()
    step_events = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
                   for _ in range(args.steps)]
    t0 = torch.cuda.Event(enable_timing=True)
    t1 = torch.cuda.Event(enable_timing=True)
    if ws > 1:
        dist.barrier()
    torch.cuda.synchronize()
    with ClockSampler(local) as clocks:
        t0.record(stream)
        for k in range(args.steps):
            one_step(step_events[k])
        t1.record(stream)
        torch.cuda.synchronize()
        if ws > 1:
            dist.barrier()
    elapsed_ms = t0.elapsed_time(t1)
    kernel_ms = sum(a.elapsed_time(b) for a, b in step_events) / (args.steps * LB_STEPS_PER_STEP)
    elapsed_ms, kernel_ms = max_over_ranks([elapsed_ms, kernel_ms], device="cuda")
    total_sites = sites * LB_STEPS_PER_STEP * args.steps * ws
    mlups = total_sites / (elapsed_ms * 1e-3) / 1e6

    # end to end through the C ABI with host buffers: populations in from pinned host
    # memory, 100 steps, diagnostics back to the host, every step.  FP32 host buffers
    # (the storage precision of the measured workload; 16-bit storage takes them too):
    # half the bytes of the float64 entry point.  Pipelined: a step's upload runs on
    # the handle's copy stream while the previous step computes, and a step's
    # diagnostics are read while the next one runs; every copy is inside the timed
    # region (the last result is read before the clock stops).
    host = torch.empty((2, 9, args.ny, args.nx), dtype=torch.float32, pin_memory=True).numpy()
    solver.populations(out=host)

    def e2e_run(n):
        solver.set_populations_async(host)
        solver.step(LB_STEPS_PER_STEP)
        solver.diagnostics_async()
        for _ in range(n - 1):
            solver.set_populations_async(host)
            solver.step(LB_STEPS_PER_STEP)
            solver.diagnostics_wait()
            solver.diagnostics_async()
        solver.diagnostics_wait()

    e2e_run(2)
    e2e_steps = max(3, args.steps // 2)
    torch.cuda.synchronize()
    if ws > 1:
        dist.barrier()
    w0 = time.perf_counter()
    e2e_run(e2e_steps)
    torch.cuda.synchronize()
    e2e_s = time.perf_counter() - w0
    (e2e_s,) = max_over_ranks([e2e_s], device="cuda")
    e2e_mlups = sites * LB_STEPS_PER_STEP * e2e_steps * ws / e2e_s / 1e6
    nrows = args.ny - 2 * params["crop_rows"]
    solver.close()

    if rank != 0:
        if ws > 1:
            dist.destroy_process_group()
        return
    peak, peak_kind = measured_peak_hbm()
    bytes_per_launch = BYTES_PER_SITE[args.storage] * sites
    achieved = bytes_per_launch / (kernel_ms * 1e-3) / 1e9
    kname = {"fused": "step_fused_kernel", "staged": "step_block_kernel", "warp": "step_warp_kernel",
             "pipe": "step_pipe_kernel", "two_pass": "collide_kernel", "decoupled": "step_dec_kernel",
             "paired": "step_pair_kernel"}[args.kernel]
    if args.kernel == "staged" and args.storage != "f32":
        kname = "step_pair_kernel"   # the block-staged kernel's default tile for 16-bit storage
    traffic = profiled_traffic(f"{kname}:{args.storage}", args.nx, args.ny)
    out = {
        "metric": METRIC, "value": round(mlups, 1), "unit": "MLUPS", "n_gpus": ws,
        "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": round(elapsed_ms / args.steps, 4), "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": args.storage, "data": "synthetic",
        "config": config_of(args, ws),
        "roofline": {"bound": "hbm", "achieved": round(achieved, 1), "peak": peak, "unit": "GB/s",
                     "frac": round(achieved / peak, 4), "traffic": traffic,
                     "kernel": kname, "algorithmic_bytes_per_launch": bytes_per_launch,
                     "launch_ms": round(kernel_ms, 5), "peak_source": f"{peak_kind} hbm_gbs"},
        "e2e": {"value": round(e2e_mlups, 1), "unit": "MLUPS",
                "h2d_bytes_per_step": 18 * sites * 4,
                "d2h_bytes_per_step": (15 + nrows) * 8 + 4},
        "gpu_launches": launches_per_step * args.steps,
        "clocks": clocks.summary(),
    }
    if ws == 1 and not args.no_extra_lines and (args.nx, args.ny) == (1024, 2048):
        # the full-size grid (10000 x 5000) in FP32 and in FP16 storage, same kernels and
        # timing (100 LB steps + diagnostics per bench step): the size at which storage
        # types are compared
        out["full_size"] = {st: grid_line(args, 10000, 5000, st) for st in ("f32", "f16")}
    if not args.no_cpu_baseline and ws == 1:
        out["cpu_baseline"] = cpu_baseline(args, budget_s=args.cpu_seconds)
    print(json.dumps(out), flush=True)
    if ws > 1:
        dist.destroy_process_group()


def grid_line(args, nx, ny, storage, steps=3, warmup=3):
    """MLUPS and HBM-roofline fraction of the step kernel on an nx x ny grid with the
    bench step of run_ours (100 LB steps + one diagnostics evaluation), CUDA events on
    the solver's stream."""
    import torch

    from paper_2101_04847_gb300 import lbm

    params = workload(args)
    params.update(nx=nx, ny=ny, seed=1)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        s = lbm.Solver(storage=storage, kernel=args.kernel, tile_y=args.tile_y, **params)
    for _ in range(warmup):
        s.step(LB_STEPS_PER_STEP)
        s.diagnostics()
    torch.cuda.synchronize()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t0.record(stream)
    for a, b in ev:
        a.record(stream)
        s.step(LB_STEPS_PER_STEP)
        b.record(stream)
        s.diagnostics()
    t1.record(stream)
    torch.cuda.synchronize()
    s.close()
    total_ms = t0.elapsed_time(t1)
    kernel_ms = sum(a.elapsed_time(b) for a, b in ev) / (steps * LB_STEPS_PER_STEP)
    peak, _ = measured_peak_hbm()
    frac = BYTES_PER_SITE[storage] * nx * ny / (kernel_ms * 1e-3) / 1e9 / peak
    return {"value": round(nx * ny * LB_STEPS_PER_STEP * steps / (total_ms * 1e-3) / 1e6, 1), "unit": "MLUPS",
            "roofline_frac": round(frac, 4), "launch_ms": round(kernel_ms, 5),
            "bytes_per_site": BYTES_PER_SITE[storage], "steps": steps, "warmup": warmup}


def _splitmix64(state: int):
    state = (state + 0x9E3779B97F4A7C15) & ((1 << 64) - 1)
    z = state
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & ((1 << 64) - 1)
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & ((1 << 64) - 1)
    return state, z ^ (z >> 31)


def ensemble_members(n: int = 16, seed: int = 0) -> list[dict]:
    """Members of the batched-ensemble workload: grids drawn uniformly from
    {512x1024, 1024x2048, 2048x4096}, G from {0.0, 1.2, 1.4}, FP32 or FP16 storage,
    from splitmix64(seed); member i is seeded i + 1."""
    grids = [(512, 1024), (1024, 2048), (2048, 4096)]
    Gs = [0.0, 1.2, 1.4]
    st = seed
    out = []
    for i in range(n):
        st, a = _splitmix64(st)
        st, b = _splitmix64(st)
        st, c = _splitmix64(st)
        nx, ny = grids[a % 3]
        G = Gs[b % 3]
        d = dict(nx=nx, ny=ny, tau_A=1.0, tau_B=1.0, G=G, mass_A=1.0, mass_B=0.9, g=1e-5, n_modes=8, amp=2.0,
                 width=1.5, minority=0.0 if G == 0.0 else 0.08, crop_rows=10, seed=i + 1,
                 storage="f16" if c % 2 else "f32")
        out.append(d)
    return out


def run_ensemble(args):
    import torch

    from paper_2101_04847_gb300 import lbm

    torch.cuda.set_device(0)
    members = ensemble_members(args.ensemble)
    if args.ensemble_grid:   # every member on one grid (e.g. small grids that cannot fill the GPU alone)
        nx, ny = (int(v) for v in args.ensemble_grid.lower().split("x"))
        members = [dict(m, nx=nx, ny=ny) for m in members]
    lb_steps = 50   # one captured 50-step graph per bench step
    params = [lbm.default_params(kernel="staged", **m) for m in members]
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ens = lbm.Ensemble(params, stream=stream.cuda_stream)
    tile_y, _ = ens.tune()
    tile_x = ens.tile_width
    for _ in range(args.warmup):
        ens.step(lb_steps)
    torch.cuda.synchronize()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with ClockSampler(0) as clocks:
        a.record(stream)
        for _ in range(args.steps):
            ens.step(lb_steps)
        b.record(stream)
        torch.cuda.synchronize()
    ens.sync()
    ens_ms = a.elapsed_time(b)
    ens.close()
    sites = sum(m["nx"] * m["ny"] for m in members)
    agg = sites * lb_steps * args.steps / (ens_ms * 1e-3) / 1e6
    # the same realisations advanced one after another, each with its own solver
    seq_ms = 0.0
    for m in members:
        with torch.cuda.stream(stream):
            s = lbm.Solver(lbm.default_params(kernel="staged", **m))   # each run with its own default tiling
        for _ in range(args.warmup):
            s.step(lb_steps)
        torch.cuda.synchronize()
        a.record(stream)
        for _ in range(args.steps):
            s.step(lb_steps)
        b.record(stream)
        torch.cuda.synchronize()
        seq_ms += a.elapsed_time(b)
        s.close()
    seq = sites * lb_steps * args.steps / (seq_ms * 1e-3) / 1e6
    bytes_per_update = sum(m["nx"] * m["ny"] * BYTES_PER_SITE[m["storage"]] for m in members)
    peak, peak_kind = measured_peak_hbm()
    achieved = bytes_per_update * lb_steps * args.steps / (ens_ms * 1e-3) / 1e9
    out = {
        "metric": METRIC, "value": round(agg, 1), "unit": "MLUPS", "n_gpus": 1, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": round(ens_ms / args.steps, 4), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32+f16", "data": "synthetic",
        "config": {"workload": f"ensemble of {len(members)} realisations, grids "
                               + (f"all {args.ensemble_grid}" if args.ensemble_grid
                                  else "from 512x1024/1024x2048/2048x4096")
                               + ", G from 0/1.2/1.4, FP32 or FP16 storage, one launch per LB step",
                   "members": [f"{m['nx']}x{m['ny']} G={m['G']} {m['storage']}" for m in members],
                   "lb_steps_per_step": lb_steps, "tile_y": tile_y, "tile_x": tile_x,
                   "l2": l2_note(bytes_per_update // 2)},
        "sequential": {"value": round(seq, 1), "unit": "MLUPS", "speedup": round(agg / seq, 3)},
        "roofline": {"bound": "hbm", "achieved": round(achieved, 1), "peak": peak, "unit": "GB/s",
                     "frac": round(achieved / peak, 4), "traffic": None, "kernel": "ensemble_step_kernel",
                     "peak_source": f"{peak_kind} hbm_gbs"},
        "gpu_launches": lb_steps * args.steps,
        "clocks": clocks.summary(),
    }
    print(json.dumps(out), flush=True)


def run_storage_study(args):
    """The same realisation advanced with FP32, FP16 and BF16 population storage; the
    16-bit runs' diagnostics are compared with the FP32 run's at checkpoints (the FP32
    path matches the FP64 oracle to ~3e-6 on the small grid, and the oracle is out of
    reach at this size).  Each storage's rate and roofline fraction are timed too."""
    import torch

    from paper_2101_04847_gb300 import lbm

    torch.cuda.set_device(0)
    params = workload(args)
    params["seed"] = 1
    total = args.storage_study
    nchk = 5
    chunk = max(1, total // nchk)
    budget = ("flux_pb", "flux_K", "flux_tau", "viscous", "buoyancy")
    keys = ("E_k", "E_p", "h", "L_int", "viscous", "enstrophy", "mass_A", "mass_B") + budget
    series, rates = {}, {}
    stream = torch.cuda.Stream()
    for storage in ("f32", "f16", "bf16"):
        with torch.cuda.stream(stream):
            s = lbm.Solver(storage=storage, kernel=args.kernel, tile_y=args.tile_y, **params)
        s.step(LB_STEPS_PER_STEP)   # warm-up of the graphs
        s.reset()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        ms = 0.0
        rows = []
        for _ in range(nchk):
            a.record(stream)
            s.step(chunk)
            b.record(stream)
            torch.cuda.synchronize()
            ms += a.elapsed_time(b)
            d = s.diagnostics(check=False)
            rows.append({k: float(d[k]) for k in keys} | {"status": int(d["status"])})
        s.close()
        series[storage] = rows
        mlups = args.nx * args.ny * chunk * nchk / (ms * 1e-3) / 1e6
        rates[storage] = {"MLUPS": round(mlups, 1), "launch_ms": round(ms / (chunk * nchk), 5),
                          "roofline_frac": round(BYTES_PER_SITE[storage] * mlups * 1e6 / 1e9 / measured_peak_hbm()[0], 4)}
    errors = {}
    for storage in ("f16", "bf16"):
        per = []
        for ref, got in zip(series["f32"], series[storage]):
            scale = max(abs(ref[k]) for k in budget)
            per.append({k: round(abs(got[k] - ref[k]) / (scale if k in budget else max(abs(ref[k]), 1e-300)), 6)
                        for k in keys})
        errors[storage] = per
    out = {"kind": "storage_study", "workload": config_of(args, 1)["workload"], "steps": chunk * nchk,
           "checkpoints": [chunk * (i + 1) for i in range(nchk)], "rates": rates,
           "relative_error_vs_f32": errors,
           "f32_series": series["f32"],
           "note": "budget terms relative to the largest budget term at that checkpoint"}
    print(json.dumps(out), flush=True)


# The paper's production case (Section 2, parameter paragraph): tau = 0.53 (nu = 0.01),
# pure densities 1.10, g = 9e-6, 10000 x 5000, 90 000 steps; G_AB = 0.1381 (immiscible)
# or 0.0805 (miscible).  Both start, as the paper's runs do, from the immiscible model's
# equilibrium configuration: each phase holds the coexistence fraction 6.8 % of the
# other component (pure phases would put the absent component 0.3 % below zero within
# a few steps of the over-relaxed BGK update at tau = 0.53).  The white-noise interface deformation of amplitude 4 is
# read as seeded sinusoidal modes normalised to amplitude 4, one mode per 128 columns
# up to 64 (at 10000 columns: wavelengths of 156 cells and more; shorter waves than
# the interface is wide drive the densities negative in the first steps).
PAPER_CASE = dict(tau_A=0.53, tau_B=0.53, mass_A=1.1, mass_B=1.1, g=9e-6, amp=4.0, width=1.5, crop_rows=10)
PAPER_COUPLING = {"immiscible": dict(G=0.1381, minority=0.068), "miscible": dict(G=0.0805, minority=0.068)}
# tension in the interface-energy relation (Section 3, Eq. "Korteweg stress and total
# length"): the Korteweg stress P^K's part of the flat interface's stress excess in the
# FP64 oracle at this coupling and reading, 0.0040 (the whole mechanical tension, which
# the Laplace law of droplets confirms, is 0.0046; the paper quotes 0.0059)
PAPER_GAMMA = 0.0040
PAPER_TERMS = ("E_k", "E_p", "h", "L_int", "buoyancy", "flux_pb", "flux_K", "flux_tau", "viscous", "enstrophy",
               "mass_A", "mass_B")


def run_paper_case(args):
    """Seeded realisations of the paper's production case advanced together through the
    ensemble API, diagnostics every `every` steps; FP32 and (paired seeds) FP16 storage.
    Prints one JSON line: ensemble mean and standard deviation of each diagnostic, the
    interface-energy relation <(div P^K) . u> against (1/D) d(gamma L)/dt, the time at
    which the interface-energy variation peaks, and the FP16-vs-FP32 error per diagnostic."""
    import numpy as np
    import torch

    from paper_2101_04847_gb300 import lbm

    torch.cuda.set_device(0)
    total, every = args.paper_case, args.paper_every
    nchk = total // every
    cases = [c.strip() for c in args.paper_cases.split(",") if c.strip()]
    stream = torch.cuda.Stream()
    results, rates = {}, {}
    for case in cases:
        coupling, storage = case.split(":")
        seeds = list(range(1, args.paper_seeds + 1))
        params = [lbm.default_params(nx=args.nx, ny=args.ny, seed=sd, storage=storage,
                                     n_modes=max(1, min(64, args.nx // 128)),
                                     **PAPER_CASE, **PAPER_COUPLING[coupling]) for sd in seeds]
        with torch.cuda.stream(stream):
            ens = lbm.Ensemble(params, stream=stream.cuda_stream)
        # a member whose guard trips (a non-finite density, or one below -5 % of rho0)
        # leaves the statistics from that checkpoint on (its values are NaN there)
        unstable = [None] * len(seeds)

        def record(ds, step):
            row = []
            for m, d in enumerate(ds):
                if unstable[m] is None and int(d["status"]) != 0:
                    unstable[m] = step
                bad = unstable[m] is not None
                row.append({k: float("nan") if bad else float(v) for k, v in d.items() if k in PAPER_TERMS})
            return row

        series = [record(ens.diagnostics(check=False), 0)]
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        ms = 0.0
        done = 0
        with ClockSampler(0) as clocks:
            for k in range(nchk):
                a.record(stream)
                ens.step(every)
                b.record(stream)
                torch.cuda.synchronize()
                ms += a.elapsed_time(b)
                done = every * (k + 1)
                series.append(record(ens.diagnostics(check=False), done))
                if all(u is not None for u in unstable):
                    break
        ens.close()
        rates[case] = {"MLUPS": round(args.nx * args.ny * len(seeds) * done / (ms * 1e-3) / 1e6, 1),
                       "seconds": round(ms / 1e3, 1), "clocks": clocks.summary(), "steps_done": done,
                       "unstable_at_step": unstable}
        results[case] = series
        if args.paper_out:   # the raw series so far, in case a later case does not finish
            Path(args.paper_out + ".partial").write_text(json.dumps({"rates": rates, "series": results}))
    steps = [every * i for i in range(nchk + 1)]
    sub = args.nx * (args.ny - 2 * PAPER_CASE["crop_rows"])
    out = {"kind": "paper_case", "grid": f"{args.nx}x{args.ny}", "steps": total, "every": every,
           "seeds": args.paper_seeds, "params": dict(PAPER_CASE, n_modes=max(1, min(64, args.nx // 128))),
           "couplings": PAPER_COUPLING,
           "gamma": PAPER_GAMMA, "rates": rates, "checkpoints": steps, "cases": {}}
    for case, series in results.items():
        while len(series) < nchk + 1:   # a case whose members all turned unstable stopped early
            series.append([{k: float("nan") for k in PAPER_TERMS} for _ in series[0]])
        arr = {k: np.array([[row[m][k] for m in range(len(row))] for row in series]) for k in PAPER_TERMS}
        with np.errstate(all="ignore"):
            stats = {k: {"mean": np.nanmean(arr[k], axis=1).tolist(), "std": np.nanstd(arr[k], axis=1).tolist(),
                         "members": np.sum(np.isfinite(arr[k]), axis=1).tolist()} for k in PAPER_TERMS}
        entry = {"series": stats}
        if case.startswith("immiscible"):
            # Section 3, Eq. "Korteweg stress and total length": <(div P^K) . u> = (1/D) d(gamma L)/dt,
            # the time derivative a centred difference of the length series
            L = arr["L_int"]
            dLdt = np.full_like(L, np.nan)
            dLdt[1:-1] = (L[2:] - L[:-2]) / (2.0 * every)
            rhs = PAPER_GAMMA * dLdt / sub
            fk = arr["flux_K"]
            with np.errstate(all="ignore"):
                mean_rhs, mean_fk = np.nanmean(rhs, axis=1), np.nanmean(fk, axis=1)
            ok = np.isfinite(mean_rhs) & np.isfinite(mean_fk)
            idx = np.where(ok & (np.array(steps) >= 10000))[0]
            corr = float(np.corrcoef(mean_fk[idx], mean_rhs[idx])[0, 1]) if len(idx) > 2 else None
            ratio = float(np.sum(mean_fk[idx] * mean_rhs[idx]) / np.sum(mean_rhs[idx] ** 2)) if len(idx) > 2 else None
            peak = int(steps[int(np.nanargmax(np.where(ok, mean_rhs, -np.inf)))])
            entry["interface_energy"] = {"rhs_mean": [None if not np.isfinite(v) else float(v) for v in mean_rhs],
                                         "flux_K_mean": mean_fk.tolist(), "correlation_after_10000": corr,
                                         "flux_over_rhs_after_10000": ratio, "peak_step_of_d_gammaL_dt": peak}
        out["cases"][case] = entry
    # FP16 against FP32 on the same seeds: relative error of the ensemble means, and the
    # median over seeds of each realisation's relative error, per checkpoint
    for coupling in PAPER_COUPLING:
        a32, a16 = results.get(f"{coupling}:f32"), results.get(f"{coupling}:f16")
        if a32 is None or a16 is None:
            continue
        err = {}
        for k in PAPER_TERMS:
            x = np.array([[r[k] for r in row] for row in a32])
            y = np.array([[r[k] for r in row] for row in a16])
            scale = np.maximum(np.abs(x), 1e-300)
            with np.errstate(all="ignore"):
                mx, my = np.nanmean(x, axis=1), np.nanmean(y, axis=1)
                err[k] = {"mean_rel": (np.abs(my - mx) / np.maximum(np.abs(mx), 1e-300)).tolist(),
                          "median_seed_rel": np.nanmedian(np.abs(y - x) / scale, axis=1).tolist()}
        out[f"{coupling}_f16_vs_f32"] = err
    if args.paper_out:
        Path(args.paper_out).write_text(json.dumps(out))
    summary = {k: v for k, v in out.items() if k not in ("cases",) and not k.endswith("_f16_vs_f32")}
    sig = lambda v: float(f"{v:.6g}")
    summary["final"] = {case: {k: [sig(out["cases"][case]["series"][k]["mean"][-1]),
                                   sig(out["cases"][case]["series"][k]["std"][-1])]
                               for k in ("h", "E_k", "E_p", "L_int")} for case in out["cases"]}
    for case in out["cases"]:
        if "interface_energy" in out["cases"][case]:
            ie = out["cases"][case]["interface_energy"]
            summary.setdefault("interface_energy", {})[case] = {k: ie[k] for k in
                                                               ("correlation_after_10000", "flux_over_rhs_after_10000",
                                                                "peak_step_of_d_gammaL_dt")}
    print(json.dumps(summary), flush=True)


def _oracle_replica(job):
    """One process of the CPU baseline: the FP64 numpy oracle as it stands, advancing its
    own replica of the workload one full-grid LB step at a time for about `budget_s`
    seconds; returns (steps, wall seconds, CPU seconds)."""
    params, budget_s = job
    from oracle import lbm_oracle as O

    p = O.Params(**params)
    f = O.step(O.initial_populations(p), p, 1)   # warm-up
    n = 0
    t, c = time.perf_counter(), time.process_time()
    while True:
        f = O.step(f, p, 1)
        n += 1
        if time.perf_counter() - t > budget_s and n >= 2:
            break
    return n, time.perf_counter() - t, time.process_time() - c


def host_workers(bytes_per_replica: float) -> int:
    """Replicas the host can run at once: one per core, as many as fit in half the
    physical memory."""
    cores = len(os.sched_getaffinity(0)) if hasattr(os, "sched_getaffinity") else (os.cpu_count() or 1)
    try:
        mem = os.sysconf("SC_PAGE_SIZE") * os.sysconf("SC_PHYS_PAGES")
    except (ValueError, OSError, AttributeError):
        mem = 0
    fit = int(0.5 * mem // bytes_per_replica) if mem else cores
    return max(1, min(cores, fit))


def cpu_baseline(args, budget_s: float, workers: int | None = None) -> dict:
    """The FP64 numpy oracle as it stands on the host's cores: independent replicas of
    the workload, one process per core (spawned, so no GPU state is inherited), each
    advancing one full-grid LB step at a time for about `budget_s` seconds; the value
    is the sum of the replicas' rates."""
    import multiprocessing as mp

    # the oracle holds the populations and a few temporaries of the same size
    per_replica = 8.0 * 18 * args.nx * args.ny * 8
    n_work = workers or host_workers(per_replica)
    jobs = [(workload(args), budget_s)] * n_work
    if n_work == 1:
        res = [_oracle_replica(jobs[0])]
    else:
        with mp.get_context("spawn").Pool(n_work) as pool:
            res = pool.map(_oracle_replica, jobs)
    rate = sum(args.nx * args.ny * n / dt for n, dt, _ in res) / 1e6
    steps = sum(n for n, _, _ in res)
    wall = max(dt for _, dt, _ in res)
    cpu = sum(c for _, _, c in res)
    return {"value": round(rate, 3), "unit": "MLUPS", "cores": round(cpu / wall, 2), "kind": "oracle",
            "sample": f"{n_work} independent replicas of the full {args.nx}x{args.ny} grid (FP64 numpy oracle, "
                      f"one process each), {steps} LB steps in all over {wall:.1f} s wall, {cpu:.1f} s CPU"}


def run_reference(args):
    """The reference arm: the FP64 oracle as it stands on the host's cores, one process
    per replica (as many as cores and memory allow); each timed step is one LB step of
    the full grid in every replica, and the value is their summed rate."""
    ws, rank, _ = dist_env()
    if rank != 0:
        return
    import multiprocessing as mp

    per_replica = 8.0 * 18 * args.nx * args.ny * 8
    n_work = host_workers(per_replica)
    jobs = [(workload(args), args.warmup, args.steps)] * n_work
    if n_work == 1:
        res = [_oracle_steps(jobs[0])]
    else:
        with mp.get_context("spawn").Pool(n_work) as pool:
            res = pool.map(_oracle_steps, jobs)
    wall = max(dt for dt, _ in res)
    cpu = sum(c for _, c in res)
    mlups = args.nx * args.ny * args.steps * n_work / wall / 1e6
    out = {
        "metric": METRIC, "value": round(mlups, 3), "unit": "MLUPS", "n_gpus": ws, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": round(wall / args.steps * 1e3, 2), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": config_of(args, ws), "impl": "reference",
        "cpu_baseline": {"value": round(mlups, 3), "unit": "MLUPS", "cores": round(cpu / wall, 2), "kind": "oracle",
                         "sample": f"each step is 1 LB step of the full {args.nx}x{args.ny} grid in each of "
                                   f"{n_work} independent replicas (FP64 numpy oracle, one process each)"},
        "e2e": {"value": round(mlups, 3), "unit": "MLUPS", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(out), flush=True)


def _oracle_steps(job):
    """One replica of the reference arm: `warmup` untimed then `steps` timed LB steps;
    returns (wall seconds, CPU seconds) of the timed ones."""
    params, warmup, steps = job
    from oracle import lbm_oracle as O

    p = O.Params(**params)
    f = O.initial_populations(p)
    for _ in range(warmup):
        f = O.step(f, p, 1)
    t, c = time.perf_counter(), time.process_time()
    for _ in range(steps):
        f = O.step(f, p, 1)
    return time.perf_counter() - t, time.process_time() - c


def run_closure(args):
    """Throughput of the learned closure at the fine workload's size: the 2x-coarsened
    run (nx/2 x ny/2, one coarse step = four fine steps) advanced in intervals of 10
    coarse steps, corrected after each (interface order parameter + velocity / 4),
    against the plain FP32 fine solver covering the same physical time.  The network
    has untrained He-scaled weights (the kernels' cost does not depend on them); its
    accuracy is measured on the 128x256 workload by the closure tests."""
    import numpy as np
    import torch

    from paper_2101_04847_gb300 import lbm

    torch.cuda.set_device(0)
    interval, mode = 10, 4
    fine = lbm.default_params(**workload(args), seed=1)
    stream = torch.cuda.Stream()
    c = lbm.Closure(fine, interval=interval, seed=0, stream=stream.cuda_stream)
    rng = np.random.default_rng(0)
    parts = []
    for shape in ((32, 4, 3, 3), (32,), (32, 32, 3, 3), (32,), (4, 32, 3, 3), (4,)):
        if len(shape) == 4:
            parts.append(rng.normal(0.0, np.sqrt(2.0 / (shape[1] * 9)), size=shape).ravel() * (0.1 if shape[0] == 4 else 1.0))
        else:
            parts.append(np.zeros(shape))
    c.set_params(np.concatenate(parts).astype(np.float32))
    # input and output scales of the size a trained network has (densities ~0.5,
    # velocities ~1e-2, corrections ~1e-3 / 1e-4): with unit output scales the
    # untrained corrections reach the limiter and drive the coarse run unstable
    # within a hundred intervals, which then times the instability guard instead
    c.set_normalisation([0.5, 0.5, 0.0, 0.0], [0.5, 0.5, 1e-2, 1e-2], [1e-3, 1e-3, 1e-4, 1e-4])
    f_solver, c_solver = c.solvers()
    ncx, ncy = c.coarse.nx, c.coarse.ny
    cnn = lbm.Cnn(ncx, ncy, stream=stream)
    dp = torch.from_numpy(np.concatenate(parts).astype(np.float32)).cuda()
    dx = torch.randn(4, ncy, ncx, device="cuda")
    dy = torch.empty_like(dx)
    torch.cuda.synchronize()

    def timed(fn, k, reps=5):
        # median of `reps` timed blocks of k calls: one block of ~0.1 s can catch a
        # stall of the whole GPU (measured once: 4.65 ms for 3.0 ms of coarse steps)
        out = []
        for _ in range(reps):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record(stream)
            for _ in range(k):
                fn()
            b.record(stream)
            torch.cuda.synchronize()
            out.append(a.elapsed_time(b) / k)
        return float(np.median(out))

    for _ in range(args.warmup):
        c.advance(1, mode)
        c.advance(1, 0)
        cnn.infer(dp, dx, dy)
    f_solver.step(4 * interval)
    torch.cuda.synchronize()
    with ClockSampler(0) as clocks:
        # one call advances args.steps intervals (it reads the CNN status once, at the end)
        corrected = timed(lambda: c.advance(args.steps, mode), 1) / args.steps
        coarse = timed(lambda: c.advance(args.steps, 0), 1) / args.steps
        infer = timed(lambda: cnn.infer(dp, dx, dy), args.steps)
        plain = timed(lambda: f_solver.step(4 * interval), max(1, args.steps // 2))
    cnn.status()
    coarse_status = c_solver.diagnostics()["status"]
    if coarse_status != lbm.LBM_OK:
        print(f"warning: the coarse run turned unstable during the timing (status {coarse_status})", file=sys.stderr)
    fine_sites = fine.nx * fine.ny
    fine_equiv = fine_sites * 4 * interval
    out = {
        "kind": "closure",
        "coarse_status": int(coarse_status),
        "metric": "fine-equivalent MLUPS (fine sites x fine steps covered per second)",
        "unit": "MLUPS",
        "value": fine_equiv / (corrected * 1e-3) / 1e6,
        "higher_is_better": True,
        "dtype": "f32 populations, bf16 CNN activations",
        "data": "synthetic",
        "config": {"workload": f"fine {fine.nx}x{fine.ny} / coarse {ncx}x{ncy} two-component D2Q9 Shan-Chen "
                               f"Rayleigh-Taylor, G=1.4, interval {interval} coarse steps, correction mode {mode}",
                   "weights": "untrained (He-scaled), output scales 1e-3 / 1e-4; throughput only"},
        "ms_per_interval": {"coarse_steps": coarse, "coarse_steps_and_correction": corrected,
                            "correction": corrected - coarse, "cnn_inference": infer,
                            "plain_fine_steps": plain},
        "plain_fine_MLUPS": fine_equiv / (plain * 1e-3) / 1e6,
        "speedup_vs_plain_fine": plain / corrected,
        "steps": args.steps, "warmup": args.warmup,
        "accuracy": "measured on 128x256 fine / 64x128 coarse (tests/test_gpu_closure.py), not at this size",
        "clocks": clocks.summary(),
    }
    c.close()
    print(json.dumps(out), flush=True)


def run_closure_accuracy(args):
    """Accuracy of the learned closure on the fine grid --nx x --ny: the regime of the
    closure tests (equal pure densities, g = 3e-4, 4-cell perturbation), trained on 6
    seeded fine runs (8 intervals of 10 coarse steps after 200 fine steps), then the
    coarse run of 3 held-out seeds over --closure-intervals intervals (default 12),
    without correction (0), with the
    order-parameter correction everywhere (3) and on the interface only (4): relative
    RMS error of h, E_k, E_p, L_int and of the kinetic-energy budget terms (viscous,
    buoyancy, bulk-pressure and Korteweg fluxes) against the fine run.  Under the
    diffusive scaling a coarse cell is twice as large (lengths 1/2) and a coarse step
    four fine steps: energies per mass scale by 4, their rates (the budget terms,
    per time step) by 16."""
    import numpy as np
    import torch

    from paper_2101_04847_gb300 import lbm

    torch.cuda.set_device(0)
    fine = lbm.default_params(nx=args.nx, ny=args.ny, tau_A=1.0, tau_B=1.0, G=1.4, mass_A=1.0, mass_B=1.0,
                              g=3e-4, n_modes=8, amp=4.0, width=1.5, minority=0.08, crop_rows=10, seed=1)
    c = lbm.Closure(fine, interval=10, seed=0)
    t0 = time.time()
    c.generate(n_runs=args.closure_runs, seed0=11, warmup=200, intervals=8)
    loss = [c.train(epochs=1, lr=2e-3, shuffle_seed=e) for e in range(25)]
    train_s = time.time() - t0

    def errors(co, fi):
        out = {}
        for k, scale in (("h", 0.5), ("E_k", 4.0), ("E_p", 4.0), ("L_int", 0.5), ("viscous", 16.0),
                         ("buoyancy", 16.0), ("flux_pb", 16.0), ("flux_K", 16.0)):
            f = np.array([d[k] for d in fi]) * scale
            q = np.array([d[k] for d in co])
            out[k] = round(float(np.sqrt(np.mean((q - f) ** 2)) / max(np.sqrt(np.mean(f ** 2)), 1e-30)), 4)
        return out

    res = {}
    for seed in (101, 102, 103):
        res[seed] = {}
        for mode in (0, 3, 4):
            try:
                res[seed][mode] = errors(*c.evaluate(seed=seed, warmup=200, intervals=args.closure_intervals,
                                                     use_net=mode))
            except lbm.LbmError as ex:   # the corrected run turned unstable: the fine run stands
                res[seed][mode] = f"status {ex.status}"
    c.close()
    print(json.dumps({"kind": "closure_accuracy", "fine": f"{args.nx}x{args.ny}", "coarse": f"{args.nx // 2}x{args.ny // 2}",
                      "intervals": args.closure_intervals, "training_runs": args.closure_runs,
                      "train": {"loss_first": round(loss[0], 4), "loss_last": round(loss[-1], 4), "seconds": round(train_s, 1)},
                      "relative_rms_error_vs_fine": res}), flush=True)


def main():
    ap = argparse.ArgumentParser(description=__doc__, formatter_class=argparse.RawDescriptionHelpFormatter)
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=30)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--storage", choices=["f32", "f16", "bf16"], default="f32")
    ap.add_argument("--kernel", choices=["fused", "two_pass", "staged", "warp", "pipe", "decoupled", "paired"], default="staged")
    ap.add_argument("--tile-y", dest="tile_y", type=int, default=0)
    ap.add_argument("--nx", type=int, default=1024)
    ap.add_argument("--ny", type=int, default=2048)
    ap.add_argument("--cpu-seconds", type=float, default=12.0)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-extra-lines", dest="no_extra_lines", action="store_true",
                    help="skip the 10000x5000 FP32 / FP16 lines added to the default run")
    ap.add_argument("--ensemble", type=int, default=0, help="run the batched-ensemble workload with this many members")
    ap.add_argument("--ensemble-grid", dest="ensemble_grid", default="",
                    help="with --ensemble: put every member on this NXxNY grid instead of the drawn ones")
    ap.add_argument("--closure-accuracy", dest="closure_accuracy", action="store_true",
                    help="train the closure on the --nx x --ny fine grid and compare held-out coarse runs with the fine run")
    ap.add_argument("--closure-intervals", dest="closure_intervals", type=int, default=12,
                    help="with --closure-accuracy: intervals of 10 coarse steps in each held-out run")
    ap.add_argument("--closure-runs", dest="closure_runs", type=int, default=6,
                    help="seeded fine runs that provide the closure's training pairs (8 intervals each)")
    ap.add_argument("--closure", action="store_true",
                    help="time the learned closure (coarse run + correction) against the plain fine solver")
    ap.add_argument("--storage-study", dest="storage_study", type=int, default=0,
                    help="advance FP32, FP16 and BF16 storage this many LB steps and compare their diagnostics")
    ap.add_argument("--paper-case", dest="paper_case", type=int, default=0,
                    help="advance the paper's production case (tau 0.53, G 0.1381 / 0.0805) this many LB steps")
    ap.add_argument("--paper-every", dest="paper_every", type=int, default=1000)
    ap.add_argument("--paper-seeds", dest="paper_seeds", type=int, default=10)
    ap.add_argument("--paper-cases", dest="paper_cases", default="immiscible:f32,immiscible:f16",
                    help="comma-separated coupling:storage runs, coupling immiscible or miscible")
    ap.add_argument("--paper-out", dest="paper_out", default="", help="write the full series to this JSON file")
    args = ap.parse_args()
    if args.warmup < 3:
        ap.error("--warmup must be >= 3")
    if args.impl == "reference":
        run_reference(args)
    elif args.ensemble:
        run_ensemble(args)
    elif args.storage_study:
        run_storage_study(args)
    elif args.paper_case:
        run_paper_case(args)
    elif args.closure:
        run_closure(args)
    elif args.closure_accuracy:
        run_closure_accuracy(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
