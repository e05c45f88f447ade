#!/usr/bin/env python3
"""Benchmark of the fused double-MRT time step (MLUPS and fraction of the HBM roofline).

One "step" is one time step of the whole cavity (pull-stream of both lattices with the
walls, D2Q9 MRT + force, D2Q5 MRT, store, hot-wall Nusselt reduction); which kernel takes a
run and how many steps a launch does is the library's own report. The default workload is the largest single cavity,
4096 x 4096 at Ra = 1e7, Pr = 0.001, alpha = 0.1, started at rest with seeded
1e-6 noise; its two float32 population buffers (3.76 GB) are far larger than L2,
so no flush is needed between steps.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl dmrt|reference]

With N > 1 (torchrun) every rank steps its own independent cavity (weak scaling,
no collective on the data path); timing is the max over ranks. The line also
carries the same cavity split into N y-slabs, one per rank, with one halo-row
exchange per step (strong scaling).
``--impl reference`` times the FP64 CPU oracle on the host cores instead.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import re
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "MLUPS (both lattices) & % HBM roofline; batched/FP16 vs plain FP32 at Nu err≤1e-3"
UNIT = "MLUPS"
BYTES_PER_NODE_FP32 = 112  # 14 populations read + 14 written, 4 bytes each
# storage mode -> (storage, rounding); bytes moved per node and step (read + write)
STORAGES = {"fp32": (0, 0), "fp16": (1, 0), "bf16": (2, 0), "fp16_sr": (1, 1), "bf16_sr": (2, 1),
            "mixed": (3, 0), "mixed_sr": (3, 1), "theta32": (4, 0), "theta32_sr": (4, 1)}
BYTES_PER_NODE = {"fp32": 112, "fp16": 56, "bf16": 56, "fp16_sr": 56, "bf16_sr": 56, "mixed": 76,
                  "mixed_sr": 76, "theta32": 60, "theta32_sr": 60}
# Storage modes of the secondary runs, each with the kernel AUTO picks.
SECONDARY_STORAGES = ("fp16", "bf16", "fp16_sr", "bf16_sr", "mixed", "mixed_sr", "theta32", "theta32_sr")
FALLBACK_HBM_GBS = 6800.0
GATE_STEPS = 20000  # the stated length of the 4096^2 workload; the Nu gate is taken over it
NU_GATE = 1e-3
BATCH_MIN_STEPS = 2000  # batched sweeps are timed over at least this many steps
SLAB_STEPS = 200  # timed steps of the single cavity split over the ranks (N > 1)
PROFILE_SUMMARY = os.path.join(ROOT, "profiles", "step_kernel_4096x4096.json")
KERNEL_SOURCES = [os.path.join(ROOT, "paper_1601_04633_gb300", "csrc", f)
                  for f in ("lattice.cuh", "collide_pair.cuh", "step_tma.cuh", "step_march.cuh", "step_direct.cuh")]


KERNELS = {1: "dmrt::step_direct_kernel", 2: "dmrt::step_tma_kernel", 3: "dmrt::step_cluster_kernel",
           4: "dmrt::step_march_kernel", 5: "dmrt::step_band_kernel"}
ON_CHIP = (3, 5)  # the state stays on chip for a launch's steps


def steps_per_pass(run):
    """Steps that one pass over the state in memory takes, from the library's report of a run."""
    return run["steps_per_launch"] if run["kernel"] not in ON_CHIP else None


def short_launch(run):
    return {"kernel": KERNELS[run["kernel"]], **{k: run[k] for k in ("steps_per_launch", "grid", "block")}}


def compact(x):
    """Secondary results in six digits, tiles without their zeros: the line stays short
    enough for a reader that keeps only its last kilobytes."""
    if isinstance(x, float):
        return float(f"{x:.6g}")
    if isinstance(x, dict):
        return {k: {t: v for t, v in y.items() if v} if k == "tile" else compact(y) for k, y in x.items()}
    return [compact(y) for y in x] if isinstance(x, list) else x


def bytes_and_frac(bytes_per_node, per_pass, mlups):
    """Bytes per node and step, and the share of the HBM copy rate; None for a state on chip."""
    if per_pass is None:
        return {"bytes_per_node": None, "roofline_frac": None}
    b = bytes_per_node / per_pass
    return {"bytes_per_node": b, "roofline_frac": b * mlups * 1e6 / 1e9 / hbm_peak()[0]}


def workload(name):
    from paper_1601_04633_gb300 import inputs

    table = {
        "cavity_4096": inputs.cavity_4096,
        "cavity_2048": lambda: inputs.Cavity(2048, 2048, 1e7, 0.001, seed=5),
        "cavity_256": inputs.cavity_256_oscillatory,
        "cavity_64": inputs.cavity_64,
    }
    cav = table[name]()
    label = f"cavity_{cav.nx}x{cav.ny}_Ra{cav.Ra:g}_Pr{cav.Pr:g}_alpha{cav.alpha:g}"
    return cav, label


def nu_rel_dev(nu, ref):
    """Largest relative deviation of a mean-Nu history from a reference history,
    step by step: max_t |nu(t) - ref(t)| / |ref(t)|."""
    nu, ref = np.asarray(nu, np.float64), np.asarray(ref, np.float64)
    return float(np.max(np.abs(nu - ref) / np.abs(ref)))


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def kernel_hash():
    """Of the kernel sources' code: comments and layout do not count."""
    h = hashlib.sha256()
    for f in KERNEL_SOURCES:
        with open(f) as fh:
            code = re.sub(r"//[^\n]*|/\*.*?\*/", "", fh.read(), flags=re.S)
        h.update(" ".join(code.split()).encode())
    return h.hexdigest()[:16]


def hbm_peak():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as fh:
            d = json.load(fh)
        for key in ("hbm_gbs", "hbm_GBs", "hbm_copy_gbs"):
            if key in d and d[key]:
                return float(d[key]), "measured"
    except (OSError, ValueError):
        pass
    return FALLBACK_HBM_GBS, "fallback"


def ncu_traffic_per_step(nodes, run):
    """DRAM bytes per step from the committed ncu summary, scaled to ``nodes``; None if
    absent, taken on a different kernel source or of another kernel than the run's."""
    try:
        with open(PROFILE_SUMMARY) as fh:
            d = json.load(fh)
    except (OSError, ValueError):
        return None
    if d.get("kernel_source_hash") != kernel_hash() or not d["kernel"].startswith(KERNELS[run["kernel"]] + "<") \
            or d["steps_per_launch"] != run["steps_per_launch"]:
        return None
    return d["dram_bytes_per_step"] * nodes / d["nodes"]


class ClockSampler:
    """nvidia-smi samples of SM clock and throttle reasons during the timed region."""

    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device_uuid):
        self.uuid = device_uuid
        self.proc = None
        self.lines = []

    def start(self):
        cmd = ["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits", "-lms", "100"]
        if self.uuid:
            cmd += ["-i", self.uuid]
        try:
            self.proc = subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
        time.sleep(0.3)

    def stop(self):
        if not self.proc:
            return
        self.proc.terminate()
        try:
            out, _ = self.proc.communicate(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
            out, _ = self.proc.communicate()
        self.lines = [l for l in out.splitlines() if l.strip()]

    def summary(self):
        rows = []
        for l in self.lines:
            parts = [p.strip() for p in l.split(",")]
            if len(parts) < 8:
                continue
            try:
                rows.append((float(parts[0]), float(parts[1]), parts[4:8]))
            except ValueError:
                continue
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no nvidia-smi samples"], "samples": 0}
        names = ("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap")
        reasons = sorted({names[i] for _, _, r in rows for i, v in enumerate(r) if v.lower().startswith("active")})
        return {"sm_mhz": statistics.median(r[0] for r in rows), "sm_max_mhz": max(r[1] for r in rows),
                "reasons": reasons, "samples": len(rows)}


def time_oracle(cav, budget_s, max_steps=50, rows=None):
    """MLUPS of the FP64 oracle on the host cores: steps of the same cavity (or of a
    band of ``rows`` rows of it) until about ``budget_s`` seconds of work."""
    import oracle as O

    threads = O.set_threads(len(os.sched_getaffinity(0)))
    ny = rows or cav.ny
    m = O.derive(cav.nx, ny, cav.Ra, cav.Pr, cav.alpha)
    from paper_1601_04633_gb300 import inputs

    th = inputs.Cavity(cav.nx, ny, cav.Ra, cav.Pr, cav.alpha, seed=cav.seed).theta0()
    f, g = O.init(m, th)
    t0 = time.perf_counter()
    O.run(m, 1, f, g)
    t1 = time.perf_counter() - t0
    steps = int(max(1, min(max_steps, budget_s / max(t1, 1e-9))))
    t0 = time.perf_counter()
    O.run(m, steps, f, g)
    dt = time.perf_counter() - t0
    out = {"value": cav.nx * ny * steps / dt / 1e6, "unit": UNIT, "cores": threads, "kind": "oracle",
           "sample": f"{steps} fp64 oracle steps of {cav.nx}x{ny} (same Ra, Pr, alpha), {dt:.1f} s"}
    # The same oracle on one thread (identical results), on a band of rows sized
    # for about a quarter of the budget.
    O.set_threads(1)
    band = max(4, min(ny, int(0.25 * budget_s / max(t1 * threads, 1e-9) * ny)))
    m1 = O.derive(cav.nx, band, cav.Ra, cav.Pr, cav.alpha)
    f1, g1 = O.init(m1, th[:band])
    t0 = time.perf_counter()
    O.run(m1, 1, f1, g1)
    dt1 = time.perf_counter() - t0
    out["single_thread"] = {"value": cav.nx * band / dt1 / 1e6, "unit": UNIT, "cores": 1,
                            "sample": f"1 fp64 oracle step of {cav.nx}x{band}, {dt1:.1f} s"}
    O.set_threads(threads)
    return out


def run_reference(args):
    ws, rank, _ = dist_env()
    if rank != 0:
        return 0
    cav, label = workload(args.workload)
    import oracle as O

    threads = O.set_threads(len(os.sched_getaffinity(0)))
    # Each step: one oracle time step of a band of the cavity sized so that the whole
    # warmup + steps run stays within a couple of minutes.
    budget_per_step = max(0.005, 120.0 / max(1, args.steps + args.warmup))
    probe_rows = 64
    m = O.derive(cav.nx, probe_rows, cav.Ra, cav.Pr, cav.alpha)
    f, g = O.init(m, np.zeros((probe_rows, cav.nx)))
    t0 = time.perf_counter()
    O.run(m, 2, f, g)
    rate = cav.nx * probe_rows * 2 / (time.perf_counter() - t0)
    rows = int(max(4, min(cav.ny, budget_per_step * rate / cav.nx)))
    m = O.derive(cav.nx, rows, cav.Ra, cav.Pr, cav.alpha)
    from paper_1601_04633_gb300 import inputs

    th = inputs.Cavity(cav.nx, rows, cav.Ra, cav.Pr, cav.alpha, seed=cav.seed).theta0()
    f, g = O.init(m, th)
    O.run(m, args.warmup, f, g)
    t0 = time.perf_counter()
    O.run(m, args.steps, f, g)
    dt = time.perf_counter() - t0
    value = cav.nx * rows * args.steps / dt / 1e6
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * dt / max(args.steps, 1),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic", "config": {"workload": label, "sample_rows": rows},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": threads, "kind": "oracle",
                         "sample": f"each step: one fp64 oracle step of {cav.nx}x{rows} rows of the cavity"},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


def slab_split_run(D, dist, cav, rank, ws, args, stream):
    """One cavity split into ws y-slabs (one per rank), SLAB_STEPS timed steps."""
    import torch

    from paper_1601_04633_gb300 import slabs

    try:
        p = D.make_params(cav.nx, cav.ny, cav.Ra, cav.Pr, cav.alpha, nu_capacity=SLAB_STEPS + args.warmup)
        run = slabs.DistributedSlab(dist, p, rank, ws, theta0=cav.theta0())
        run.step(args.warmup)
        torch.cuda.synchronize()
        dist.barrier()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        run.step(SLAB_STEPS)
        e1.record(stream)
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1)
        run.slab.check()
        series = run.nusselt_series(SLAB_STEPS)
        run.close()
        t = torch.tensor([ms], dtype=torch.float64, device="cuda")
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        ms = t.item()
        return {"value": cav.nx * cav.ny * SLAB_STEPS / (ms / 1e3) / 1e6, "unit": UNIT, "scaling": "strong",
                "ranks": ws, "steps": SLAB_STEPS, "ms_per_step": ms / SLAB_STEPS,
                "nu_mean_last": float(series[-1]),
                "workload": f"one {cav.nx}x{cav.ny} cavity in {ws} y-slabs, one halo-row exchange per step"}
    except Exception as exc:  # reported on the line; the headline stands on its own
        return {"error": f"{type(exc).__name__}: {exc}"}


def run_dmrt(args):
    import torch

    ws, rank, local = dist_env()
    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device (there is no CPU fallback)")
    torch.cuda.set_device(local)
    dist = None
    if ws > 1:
        import torch.distributed as dist

        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    import __graft_entry__

    if rank == 0:
        __graft_entry__.build()
    if dist:
        dist.barrier()
    from paper_1601_04633_gb300 import dmrt as D
    from paper_1601_04633_gb300 import inputs

    cav, label = workload(args.workload)
    cav.seed = cav.seed + 1000 * rank  # independent replica per rank
    nodes = cav.nx * cav.ny
    stream = torch.cuda.current_stream()

    kw = dict(kernel=args.kernel, tma_rows=args.tma_rows, tma_stages=args.tma_stages,
              tma_npt=args.tma_npt, storage=STORAGES[args.storage][0], rounding=STORAGES[args.storage][1])
    sim = D.Cavity2D.from_inputs(cav, nu_capacity=max(args.steps + args.warmup, 1), **kw)
    sim.step(args.warmup)
    sim.check()
    torch.cuda.synchronize()

    props = torch.cuda.get_device_properties(local)
    uuid = str(getattr(props, "uuid", "") or "")
    sampler = ClockSampler(("GPU-" + uuid) if uuid and not uuid.startswith("GPU-") else uuid)
    sampler.start()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    run = sim.run_launch(max(args.steps, 1))
    per_pass = steps_per_pass(run)
    ev0.record(stream)
    sim.step(args.steps)
    ev1.record(stream)
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    sampler.stop()
    ms = ev0.elapsed_time(ev1)
    sim.check()
    nu_mean, _, _ = sim.nusselt()
    sim.close()
    del sim

    # Secondary: the 16-bit and mixed storage variants on the same workload over
    # its stated 20,000 steps, each timed over the whole run, with the gate of the
    # metric: the mean-Nu history within 1e-3 (max relative deviation) of the
    # float32 run's over the same steps.
    secondary = {}
    if not args.no_secondary and args.storage == "fp32":
        gate_steps = GATE_STEPS

        def timed_run(**kw2):
            s2 = D.Cavity2D.from_inputs(cav, nu_capacity=gate_steps + args.warmup, **kw2)
            s2.step(args.warmup)
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            s2.step(gate_steps)
            e1.record(stream)
            torch.cuda.synchronize()
            ms2 = e0.elapsed_time(e1)
            s2.check()
            series2 = s2.nusselt(series_cap=gate_steps)[2]
            launch2 = s2.run_launch(gate_steps)
            s2.close()
            return ms2, series2, launch2

        ms_ref, nu_ref, _ = timed_run(**kw)
        secondary["fp32_gate_reference"] = {"value": nodes * gate_steps / (ms_ref / 1e3) / 1e6, "unit": UNIT,
                                            "steps": gate_steps, "nu_mean_last": float(nu_ref[-1])}
        for st in SECONDARY_STORAGES:
            ms2, nu2, launch2 = timed_run(storage=STORAGES[st][0], rounding=STORAGES[st][1])
            err = nu_rel_dev(nu2, nu_ref)
            v2 = nodes * gate_steps / (ms2 / 1e3) / 1e6
            secondary[st] = {"value": v2, "unit": UNIT, "steps": gate_steps,
                             "launch": short_launch(launch2),
                             **bytes_and_frac(BYTES_PER_NODE[st], steps_per_pass(launch2), v2),
                             "nu_mean_last": float(nu2[-1]),
                             "nu_max_rel_dev_vs_fp32": err, "nu_gate_ok": bool(err <= NU_GATE),
                             "vs_fp32_single": v2 / secondary["fp32_gate_reference"]["value"]}
        secondary["nu_gate"] = (f"max over the {gate_steps} steps of |Nu(t) - Nu_fp32(t)| / |Nu_fp32(t)| "
                                f"<= {NU_GATE:g}; a variant with nu_gate_ok false does not count for the metric")

    # Small cavities (state resident in L2, launch-bound): MLUPS only; the
    # roofline fraction is reported for the large cavity and the batched sweep.
    if not args.no_secondary and args.storage == "fp32":
        small = {}
        for name, cav_s, st, n_s in (("cavity_64_fp32", inputs.cavity_64(), 0, 20000),
                                     ("cavity_128_adjoint_fp32", inputs.cavity_128_adjoint(), 0, 10000),
                                     ("cavity_256_fp32", inputs.cavity_256_oscillatory(), 0, 20000),
                                     ("cavity_256_mixed", inputs.cavity_256_oscillatory(), 3, 20000),
                                     ("cavity_256_fp16", inputs.cavity_256_oscillatory(), 1, 20000),
                                     ("cavity_256_bf16", inputs.cavity_256_oscillatory(), 2, 20000)):
            s3 = D.Cavity2D.from_inputs(cav_s, nu_capacity=n_s + args.warmup, storage=st)
            s3.step(args.warmup)
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            s3.step(n_s)
            e1.record(stream)
            torch.cuda.synchronize()
            s3.check()
            ms3 = e0.elapsed_time(e1)
            small[name] = {"value": cav_s.nx * cav_s.ny * n_s / (ms3 / 1e3) / 1e6, "unit": UNIT,
                           "steps": n_s, "us_per_step": 1e3 * ms3 / n_s, "launch": short_launch(s3.run_launch(n_s))}
            s3.close()
            del s3
        secondary["small_cavities"] = small

    # Batched sweep (64 cavities of uneven sizes and (Ra, Pr)) with the autotuned
    # schedule, against the same cavities stepped one after another through their
    # own contexts. Schedules: one launch per time step over every cavity, and
    # those the tuner also tries (several steps per launch, cavities in L2-sized
    # groups); both the one-launch-per-step figure and the tuned one are
    # reported. Tuning runs before, and outside, the timed region.
    if not args.no_secondary and args.storage == "fp32":
        from paper_1601_04633_gb300 import sharding, tune

        # With N ranks the 64 cavities are split by node count (no exchange between ranks).
        full = inputs.batch_sweep()
        sweep = sharding.shard(full, rank, ws) if ws > 1 else full
        bnodes = sum(c.nx * c.ny for c in full)
        bsteps = max(args.steps, BATCH_MIN_STEPS) // 2 * 2
        peak_hbm = hbm_peak()[0]

        def run_batch(opts, storage, rounding):
            batch = D.Batch.from_inputs(sweep, opts=opts, nu_capacity=bsteps + args.warmup, storage=storage,
                                        rounding=rounding)
            run_b = batch.run_launch(bsteps)
            batch.step(max(args.warmup, 64))
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            batch.step(bsteps)
            e1.record(stream)
            torch.cuda.synchronize()
            ms_b = e0.elapsed_time(e1)
            batch.check()
            nu = [m.nusselt(series_cap=bsteps)[2] for m in batch.members]
            batch.close()
            if dist:
                tt = torch.tensor([ms_b], dtype=torch.float64, device="cuda")
                dist.all_reduce(tt, op=dist.ReduceOp.MAX)
                ms_b = tt.tolist()[0]
            return ms_b, nu, run_b

        def batch_pass(run_b, opts):
            # Several steps of a resident group (a schedule with a tile) still move a state per step.
            return run_b["steps_per_launch"] if opts["tma_npt"] <= 0 else 1

        def max_dev(xs, refs):
            return max(nu_rel_dev(a, b_) for a, b_ in zip(xs, refs))

        nu_fp32 = None
        for tag, storage, rnd, bpn in (("batched", 0, 0, 112), ("batched_mixed", 3, 0, 76),
                                       ("batched_mixed_sr", 3, 1, 76)):
            tuned = tune.tune_batch(sweep, steps=200, warmup=10, storage=storage, rounding=rnd,
                                    group_bytes=tune.GROUP_BYTES, steps_per_launch=tune.STEPS_PER_LAUNCH)
            one = [t for t in tuned["trials"] if t["opts"]["tma_npt"] > 0
                   and t["opts"].get("group_bytes", 0) == 0 and t["opts"].get("steps_per_launch", 1) <= 1]
            best_one = max(one, key=lambda t: t["mlups"])["opts"]
            ms_st, nu_st, run_best = run_batch(best_one, storage, rnd)
            v1 = bnodes * bsteps / (ms_st / 1e3) / 1e6
            entry = {"nodes": bnodes, "steps": bsteps,
                     "one_launch_per_step": {"value": v1, "unit": UNIT, "tile": best_one,
                                             "roofline_frac": bpn * v1 * 1e6 / 1e9 / peak_hbm}}
            nu_best, best_value, entry["tile"] = nu_st, v1, best_one
            if tuned["opts"] != best_one:
                ms_b2, nu_b2, run_b2 = run_batch(tuned["opts"], storage, rnd)
                v2 = bnodes * bsteps / (ms_b2 / 1e3) / 1e6
                entry["tuned_schedule"] = {"value": v2, "unit": UNIT, "tile": tuned["opts"],
                                           "launch": short_launch(run_b2),
                                           **bytes_and_frac(bpn, batch_pass(run_b2, tuned["opts"]), v2),
                                           "nu_max_rel_diff_vs_one_launch_per_step": max_dev(nu_b2, nu_st)}
                if v2 > best_value:
                    best_value, nu_best, entry["tile"], run_best = v2, nu_b2, tuned["opts"], run_b2
            entry["value"] = best_value
            entry["unit"] = UNIT
            entry.update(bytes_and_frac(bpn, batch_pass(run_best, entry["tile"]), best_value))
            # The three best of the tuner's trials (all of them would make a line of 40 KB).
            top = sorted(tuned["trials"], key=lambda t: -t["mlups"])[:3]
            entry["tuner"] = {"trials": len(tuned["trials"]),
                              "best": [{"tile": t["opts"], "mlups": round(t["mlups"])} for t in top]}
            if storage == 0:
                nu_fp32 = nu_best
                entry["workload"] = ("64 cavities, sides {128,192,256,384}, Ra log-uniform [1e4,1e6], "
                                     "Pr {0.001,0.005,0.01}, alpha 0.1"
                                     + (f", split over {ws} ranks by node count" if ws > 1 else ""))
            else:
                entry["nu_max_rel_diff_vs_float32_batch"] = max_dev(nu_best, nu_fp32)
                entry["nu_gate_ok"] = bool(entry["nu_max_rel_diff_vs_float32_batch"] <= NU_GATE)
            secondary[tag] = entry

        # The same cavities stepped one after another through their own contexts.
        seq = [D.Cavity2D.from_inputs(c, nu_capacity=bsteps + args.warmup) for c in sweep]
        for m in seq:
            m.step(args.warmup)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for m in seq:
            m.step(bsteps)
        e1.record(stream)
        torch.cuda.synchronize()
        ms_s = e0.elapsed_time(e1)
        nu_s = [m.nusselt(series_cap=bsteps)[2] for m in seq]
        for m in seq:
            m.check()
            m.close()
        del seq
        if dist:
            tt = torch.tensor([ms_s], dtype=torch.float64, device="cuda")
            dist.all_reduce(tt, op=dist.ReduceOp.MAX)
            ms_s = tt.tolist()[0]
        secondary["batched"]["sequential_value"] = bnodes * bsteps / (ms_s / 1e3) / 1e6
        secondary["batched"]["nu_max_rel_diff_vs_sequential"] = max_dev(nu_fp32, nu_s)

        # Discrete adjoint (128 x 128, Ra 1e5, Pr 0.01, hot wall 0.5 + 0.01 N(0,1), 10000 steps,
        # J = mean Nu of the last 2000): wall time against the plain forward run.
        acav = inputs.cavity_128_adjoint()
        fwd = D.Cavity2D.from_inputs(acav, nu_capacity=2000)
        fwd.step(16)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        fwd.step(10000)
        fwd.check()
        t_fwd = time.perf_counter() - t0
        fwd.close()
        adj = D.Cavity2D.from_inputs(acav, nu_capacity=2000)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        Jv, dth, dRa = adj.adjoint(10000, 2000, store="all")
        t_adj = time.perf_counter() - t0
        adj.close()
        secondary["adjoint"] = {"workload": "cavity 128x128 Ra 1e5 Pr 0.01, 10000 steps, J over last 2000",
                                "store": "every forward state",
                                "forward_s": t_fwd, "adjoint_s": t_adj, "ratio": t_adj / t_fwd,
                                "J": Jv, "dJ_dRa": dRa, "dJ_dthetaw_norm": float(np.linalg.norm(dth))}

    # With N > 1 ranks: one cavity of the same workload split into N y-slabs, one
    # per rank, with one halo-row exchange per step over NCCL (strong scaling),
    # beside the independent replicas of the headline.
    if dist and not args.no_secondary:
        secondary["slab_split"] = slab_split_run(D, dist, cav, rank, ws, args, stream)

    # End to end through the public C ABI with host buffers: create from a pinned
    # host temperature field (H2D), K steps, then the Nu series and the u, v, theta
    # fields back to pinned host memory (D2H), all inside the timed region.
    theta0 = torch.from_numpy(cav.theta0()).pin_memory()
    outs = [torch.empty((cav.ny, cav.nx), dtype=torch.float32).pin_memory() for _ in range(3)]
    p = D.make_params(cav.nx, cav.ny, cav.Ra, cav.Pr, cav.alpha, nu_capacity=max(args.steps, 1), **kw)
    wsb = D.dmrt_workspace_size(p)
    workspace = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    series = np.zeros(max(args.steps, 1))
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    t0 = time.perf_counter()
    h = D.dmrt_create(p, theta0.numpy(), workspace.data_ptr(), wsb, stream.cuda_stream)
    D.dmrt_step(h, args.steps)
    _, _, series = D.dmrt_nusselt(h, cav.ny, args.steps)
    D.dmrt_fields(h, outs[0].data_ptr(), outs[1].data_ptr(), outs[2].data_ptr(), False)
    e2e_s = time.perf_counter() - t0
    D.dmrt_destroy(h)
    del workspace

    t = torch.tensor([ms, e2e_s], dtype=torch.float64, device="cuda")
    if dist:
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
    ms, e2e_s = t.tolist()
    if rank != 0:
        dist.destroy_process_group()
        return 0

    steps = max(args.steps, 1)
    value = ws * nodes * args.steps / (ms / 1e3) / 1e6
    per_launch_s = ms / 1e3 / steps
    peak, peak_src = hbm_peak()
    one_step = BYTES_PER_NODE[args.storage] * nodes / per_launch_s / 1e9
    if per_pass is None:
        roofline = {"bound": "latency (the state stays on chip)", "achieved": None, "peak": peak, "unit": "GB/s",
                    "frac": None, "traffic": None, "peak_source": f"{peak_src} HBM copy bandwidth",
                    "steps_per_launch": run["steps_per_launch"], "kernel": KERNELS[run["kernel"]]}
    else:
        traffic = ncu_traffic_per_step(nodes, run) if args.storage == "fp32" else None
        roofline = {"bound": "hbm", "achieved": one_step / per_pass, "peak": peak, "unit": "GB/s",
                    "frac": one_step / per_pass / peak, "traffic": traffic,
                    "peak_source": f"{peak_src} HBM copy bandwidth",
                    "bytes_per_node": BYTES_PER_NODE[args.storage] / per_pass, "steps_per_pass": per_pass,
                    "one_step_per_pass_frac": one_step / peak, "kernel": KERNELS[run["kernel"]]}
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms / steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32" if args.storage == "fp32" else f"{args.storage} storage, f32 arithmetic",
        "data": "synthetic",
        "config": {"workload": label, "nx": cav.nx, "ny": cav.ny, "Ra": cav.Ra, "Pr": cav.Pr,
                   "alpha": cav.alpha, "storage": args.storage, "parallelism": f"{ws} independent cavities",
                   "launch": short_launch(run),
                   "l2": "state (two 14-plane fp32 buffers) larger than L2: no flush"
                   if BYTES_PER_NODE[args.storage] * nodes > 129e6 else "state fits in L2"},
        "roofline": roofline,
        "e2e": {"value": ws * nodes * args.steps / e2e_s / 1e6, "unit": UNIT,
                "h2d_bytes_per_step": 8 * nodes / steps,
                "d2h_bytes_per_step": (12 * nodes + 8 * args.steps) / steps},
        "gpu_launches": run["launches"],
        "clocks": sampler.summary(),
        "nu_mean_last": nu_mean,
    }
    for tag in ("batched", "batched_mixed", "batched_mixed_sr"):
        if tag in secondary:
            secondary[tag]["vs_fp32_single"] = secondary[tag]["value"] / value
    if secondary:
        line["secondary"] = compact(secondary)
    if ws == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = time_oracle(cav, budget_s=12.0)
    print(json.dumps(line), flush=True)
    if dist:
        dist.destroy_process_group()
    return 0


def main():
    ap = argparse.ArgumentParser(description=__doc__, formatter_class=argparse.RawDescriptionHelpFormatter)
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20000)  # the 4096^2 workload is stated at 20,000 timed steps
    ap.add_argument("--warmup", type=int, default=20)
    ap.add_argument("--impl", choices=("dmrt", "reference"), default="dmrt")
    ap.add_argument("--workload", default="cavity_4096", choices=("cavity_4096", "cavity_2048", "cavity_256", "cavity_64"))
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--kernel", type=int, default=0, help="0 auto, 1 direct, 2 TMA")
    ap.add_argument("--tma-rows", type=int, default=0)
    ap.add_argument("--tma-stages", type=int, default=0)
    ap.add_argument("--tma-npt", type=int, default=0)
    ap.add_argument("--storage", choices=tuple(STORAGES), default="fp32")
    ap.add_argument("--no-secondary", action="store_true", help="skip the 16-bit storage runs")
    args = ap.parse_args()
    args.warmup = max(args.warmup, 3)
    if args.impl == "reference":
        return run_reference(args)
    return run_dmrt(args)


if __name__ == "__main__":
    sys.exit(main())
