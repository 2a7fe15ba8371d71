"""Benchmark: solves/s to max(|H|, |M_i|) <= 1e-10 on one GB300 (CUDA library via its C ABI).

Workload: periodic cube L = 32, 128^3 cells, 4th-order stencils, 6-level V-cycle,
phi = 1 + 16 seeded Fourier modes (|k| <= 4 (2 pi/L), amplitude a0/|k|, uniform
phases), Pi likewise, m = 1, K from the integrability condition.  One step is one
full solve from psi = 1, W = 0 with the sources resident on the device: FP32
inner V-cycles under FP64 defect correction (the library's MG_MIXED path).  The
same solve in plain FP64 (MG_FP64) is measured alongside for context.

Usage: python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]
N > 1 runs one independent replica per rank (instances are independent; no
collective on the data path) and reports the aggregate.
"""
import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

from paper_2501_13046_gb300 import replicas
from paper_2501_13046_gb300.replicas import dist_env

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "solves/s to |H|,|M|<=1e-10 (CTT constraints, 128^3 periodic, 4th order)"
UNIT = "solves/s"
WORKLOAD = dict(workload="periodic random-mode cosmology, L=32, 128^3, 4th-order, 6-level V-cycle, "
                         "16 modes |k|<=4(2pi/L), a0=5e-5, phi0=1, m=1, tol 1e-10",
                n=128, order=4, bc="periodic", levels=6, tol=1e-10, cells=128 ** 3)


_T0 = time.perf_counter()


def phase(name):
    """Progress of the benchmark's phases on stderr (the result line goes to stdout)."""
    print("[bench %7.1f s] %s" % (time.perf_counter() - _T0, name), file=sys.stderr, flush=True)


def peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return json.load(f), "measured"
    except OSError:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0}, "fallback"


class ClockSampler:
    """nvidia-smi clock/throttle samples during the timed region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index, self.rows, self.proc = index, [], None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), "--query-gpu=" + self.Q,
                                          "--format=csv,noheader,nounits", "-lms", "50"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except OSError:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.rows.append([c.strip() for c in line.split(",")])

    def __exit__(self, *a):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
            self.t.join(timeout=2)

    def summary(self):
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in self.rows:
            try:
                sm.append(float(r[1]))
                mx = float(r[2])
                for nm, v in zip(names, r[5:9]):
                    if v.lower() == "active":
                        reasons.add(nm)
            except (ValueError, IndexError):
                continue
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": mx, "reasons": sorted(reasons),
                "samples": len(sm)}


def fields_mod():
    from paper_2501_13046_gb300 import fields
    return fields


def make_problem():
    from paper_2501_13046_gb300 import fields
    return fields.modes_periodic(n=WORKLOAD["n"])


GOLDEN = os.path.join(ROOT, "tests", "golden")


def golden(name):
    """Sampled oracle root of a full-size workload (tests/golden/make_oracle_roots.py), or None."""
    try:
        with open(os.path.join(GOLDEN, name + "_oracle_root.json")) as f:
            return json.load(f)
    except OSError:
        return None


def oracle_iters_to(gold, tol):
    """Outer iterations the oracle needed to reach max(|H|, |M_i|) <= tol (its stored history)."""
    for it, row in enumerate(gold["oracle_history"]):
        if max(row) <= tol:
            return it
    return len(gold["oracle_history"]) - 1


def psi_background_at(gold, punctures):
    """1 + sum of m / 2r at the stored cells of a sampled oracle root."""
    cells = np.array(gold["cells"])
    n = gold["n"]
    lo = [gold["lo"]] * 3 if np.isscalar(gold["lo"]) else gold["lo"]
    hi = [gold["hi"]] * 3 if np.isscalar(gold["hi"]) else gold["hi"]
    idx = [cells % n[0], (cells // n[0]) % n[1], cells // (n[0] * n[1])]
    x = [lo[a] + (idx[a] + 0.5) * (hi[a] - lo[a]) / n[a] for a in range(3)]
    bg = np.ones(len(cells))
    for pun in punctures:
        bg += pun[0] / (2.0 * np.sqrt(sum((x[a] - pun[1][a]) ** 2 for a in range(3))))
    return bg


def field_errors(gold, u, W, psibg=None):
    """|gpu - oracle| / max |oracle field| over the stored cells, for psi, W_x, W_y, W_z (psibg: the
    puncture background at those cells, 1 without punctures)."""
    cells = np.array(gold["cells"])
    bg = 1.0 if psibg is None else psibg
    u = np.asarray(u).reshape(-1)
    W = np.asarray(W).reshape(3, -1)
    pairs = {"psi": (bg + u[cells], bg + np.array(gold["u"])), "Wx": (W[0][cells], np.array(gold["Wx"])),
             "Wy": (W[1][cells], np.array(gold["Wy"])), "Wz": (W[2][cells], np.array(gold["Wz"]))}
    return {f: float(np.abs(a - b).max() / gold["max_abs"][f]) for f, (a, b) in pairs.items()}


def cpu_model():
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.startswith("Model name"):
                return line.split(":", 1)[1].strip()
    except (OSError, subprocess.SubprocessError):
        pass
    return None


def oracle_full_size(p, threads):
    """The CPU FP64 oracle, as it stands, on the benchmarked 128^3 inputs themselves: one residual
    evaluation and one outer iteration (residual, V-cycle, update, residual) are timed, and the solve
    time is the oracle's iteration count to 1e-10 (its stored full run) times the iteration plus one
    more residual: t = (I + 1) t_res + I (t_1 - 2 t_res).  Returns (solves/s, detail)."""
    from oracle import oracle as O
    used = O.set_threads(threads)
    g = O.make_grid(p["n"], p["lo"], p["hi"], p["order"], p["bc"])
    args = (g, p["rho0"], p["rho2"], p["S"], O.K_INTEGRABILITY)
    t0 = time.perf_counter()
    O.solve(*args, tol=WORKLOAD["tol"], max_outer=0)
    t_res = time.perf_counter() - t0
    t0 = time.perf_counter()
    O.solve(*args, tol=WORKLOAD["tol"], max_outer=1)
    t_1 = time.perf_counter() - t0
    gold = golden("modes_periodic_%d" % WORKLOAD["n"])
    iters = oracle_iters_to(gold, WORKLOAD["tol"]) if gold else 14
    t_solve = (iters + 1) * t_res + iters * max(t_1 - 2 * t_res, 0.0)
    return 1.0 / t_solve, dict(threads=used, t_residual_s=t_res, t_iteration_s=t_1 - t_res, iters_to_tol=iters,
                               solve_s=t_solve)


def oracle_sample(p, seconds_budget=20.0):
    """The CPU FP64 oracle, as it stands, on a bounded sample of the workload (one step of the
    reference arm): the same field recipe and box at 32^3, solved to 1e-10, scaled to 128^3 by the
    cell count and by the ratio of the oracle's own iteration counts to 1e-10 at the two sizes
    (multigrid work per iteration is O(N); the 128^3 count is from the stored full run).
    Returns (value solves/s, detail)."""
    from oracle import oracle as O
    from paper_2501_13046_gb300 import fields
    n = 32
    q = fields.modes_periodic(n=n)
    g = O.make_grid(q["n"], q["lo"], q["hi"], q["order"], q["bc"])
    t0 = time.perf_counter()
    solves = 0
    while True:
        r = O.solve(g, q["rho0"], q["rho2"], q["S"], O.K_INTEGRABILITY, tol=WORKLOAD["tol"], max_outer=60)
        solves += 1
        if time.perf_counter() - t0 > seconds_budget / 2 or solves >= 3:
            break
    dt = (time.perf_counter() - t0) / solves
    gold = golden("modes_periodic_%d" % WORKLOAD["n"])
    it_full = oracle_iters_to(gold, WORKLOAD["tol"]) if gold else r["iters"]
    scale = (WORKLOAD["n"] / n) ** 3 * (it_full + 1) / (r["iters"] + 1)
    threads = O.set_threads(0)
    return 1.0 / (dt * scale), dict(cores=threads, sample="oracle solve of the same recipe at 32^3 (%d outer "
                                    "iterations, %.2f s per solve), scaled to 128^3 by the cell count (x64) and by the "
                                    "oracle's iteration counts to 1e-10 (%d at 128^3 in its stored full run): x%.1f"
                                    % (r["iters"], dt, it_full, scale), status=r["status"])


def run_reference(args):
    """The CPU oracle, as it stands, timed on this host on the same metric: each step is one
    bounded sample (see oracle_sample).  Under torchrun only rank 0 runs."""
    ws, rank, _ = dist_env()
    if rank != 0:
        return 0
    p = None
    for _ in range(args.warmup):
        oracle_sample(p, seconds_budget=0.0)
    times, walls, det = [], [], None
    for _ in range(args.steps):
        t0 = time.perf_counter()
        v, det = oracle_sample(p, seconds_budget=0.0)
        walls.append(time.perf_counter() - t0)
        times.append(1.0 / v)
    value = 1.0 / statistics.mean(times)
    # ms_per_step: the wall time of one step as run (one bounded sample); the 128^3 solve time the
    # sample stands for is reported beside it
    line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": statistics.mean(walls) * 1e3,
            "extrapolated_ms_per_solve": statistics.mean(times) * 1e3, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic", "impl": "reference",
            "config": WORKLOAD,
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": det["cores"], "kind": "oracle",
                             "sample": det["sample"]},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line))
    return 0


def batch_measure(mg, torch, sp, precision, repeats=1):
    """64 independent periodic instances, n drawn from {48, 64, 96, 128, 160}, a0 ~ U[2e-5, 8e-5]
    (the batched workload), solved together as one graph per round.  Returns a summary dict."""
    from paper_2501_13046_gb300 import fields
    sizes = fields.batch_sizes()
    ps = [fields.batch_instance(n, a0, seed, device="cuda") for n, a0, seed in sizes]
    cfgs = [mg.config_for(p, precision, tol=WORKLOAD["tol"], max_outer=60) for p in ps]
    # one-time tuning (untimed) on the first instance of the largest size, which dominates the
    # batch; the batch iterates in lock step until its slowest instance converges, so every
    # instance uses the same setting rather than one tuned on a single instance of its size
    big = max(range(len(ps)), key=lambda b: ps[b]["n"][0])
    pb = ps[big]
    best, tms = mg.mg_autotune(cfgs[big], pb["rho0"], pb["rho2"], pb["S"][0], pb["S"][1], pb["S"][2], stream=sp)
    tuned = {pb["n"][0]: tune_summary(best, tms)}
    for c in cfgs:
        apply_tuned(c, tuned[pb["n"][0]])
    bt = mg.mg_batch_create(cfgs, sp)
    try:
        for b, p in enumerate(ps):
            mg.mg_batch_set_sources(bt, b, p["rho0"], p["rho2"], p["S"][0], p["S"][1], p["S"][2])
        mg.mg_batch_solve(bt, len(ps))             # warm-up: captures the batch graphs
        best = None
        for _ in range(repeats):
            for b in range(len(ps)):
                mg.mg_batch_set_initial_guess(bt, b, None, None)
            st, infos, total = mg.mg_batch_solve(bt, len(ps))
            assert st == mg.MG_OK
            if best is None or total < best[2]:
                best = (st, infos, total)
    finally:
        mg.mg_batch_destroy(bt)
    st, infos, total = best
    lat = sorted(i["device_ms"] for i in infos)
    cells = sum(n ** 3 for n, _, _ in sizes)
    return {"instances": len(ps), "cells": cells, "ms": total, "solves_per_s": len(ps) / (total * 1e-3),
            "tuned": {str(k): v for k, v in sorted(tuned.items())},
            "gridpoints_per_s": cells / (total * 1e-3), "p50_ms": lat[len(lat) // 2],
            "p99_ms": lat[min(len(lat) - 1, int(0.99 * len(lat)))],
            "rounds": max(i["outer_iters"] for i in infos),
            "max_norm": max(float(i["norms"].max()) for i in infos)}


# FP64-pipe instructions of the fused residual per cell (multiply-adds, additions, conversions), from one ncu capture
# at 128^3 (3,332,789 warp instructions, profiles/outer_residual_128cube_periodic_o4.md); its stencils are 64-bit integer
# arithmetic.
RESIDUAL_FP64_PER_CELL = 50.9
# Issue slots of the FP64 pipe per second from unit counts and clocks (the denominator of an ALU-bound kernel): 152 SMs x 2
# lanes x 2.07 GHz.  A slot holds any FP64 instruction, so this is the pipe's occupancy and no rate of flops.
FP64_PEAK_TSLOTS = 152 * 2 * 2.07e9 / 1e12
# DRAM bytes of one 128^3 residual launch (dram__bytes_read.sum + dram__bytes_write.sum) from one ncu
# capture (the same file); None if none
RESIDUAL_TRAFFIC_128 = 161633536 + 56829952
# the same for the finest colour pass and residual + restriction at 128^3
# (profiles/smooth_tile_128cube_periodic_o4.md, profiles/restrict_tile_128cube_periodic_o4.md)
COLOUR_TRAFFIC_128 = 59366656 + 1694976
RESTRICT_TRAFFIC_128 = 85024512 + 2426368


def kernel_rooflines(mg, ctx, N):
    """Live CUDA-event timings (library stream) of the dominant kernel and of the colour pass."""
    pk, src = peaks()
    msb, bytesb = mg.mg_time_kernel(ctx, 2, 10)   # fused FP64 residual
    ms0, bytes0 = mg.mg_time_kernel(ctx, 0, 40)   # finest FP32 colour pass
    ms1, bytes1 = mg.mg_time_kernel(ctx, 1, 20)   # finest residual + restriction
    fp64 = mg.mg_fp64_fma_rate(ctx, 3)           # FP64 FMA rate of the library probe (context)
    ach = RESIDUAL_FP64_PER_CELL * N / (msb * 1e-3) / 1e12
    sm_gbs = bytes0 / (ms0 * 1e-3) / 1e9
    rr_gbs = bytes1 / (ms1 * 1e-3) / 1e9
    return {"bound": "alu", "achieved": ach, "peak": FP64_PEAK_TSLOTS, "unit": "1e12 FP64 issue slots/s",
            "frac": ach / FP64_PEAK_TSLOTS, "traffic": RESIDUAL_TRAFFIC_128 if N == 128 ** 3 else None,
            "kernel": "k_outer_residual<4,periodic> (fused FP64 residual, 128^3; FP64 and integer pipes)",
            "ms_per_launch": msb, "fp64_issue_slots": RESIDUAL_FP64_PER_CELL * N, "algorithmic_bytes": bytesb,
            "peak_source": "derived: 152 SMs x 2 FP64 lanes x 2.07 GHz",
            "fp64_probe_tflops": fp64, "frac_of_probe": 2 * ach / fp64,
            "colour_pass": {"bound": "hbm", "kernel": "k_smooth_tile<float,4,periodic,c> (finest, one colour)",
                            "ms_per_launch": ms0, "algorithmic_bytes": bytes0, "achieved": sm_gbs,
                            "unit": "GB/s", "peak": pk["hbm_gbs"], "frac": sm_gbs / pk["hbm_gbs"],
                            "traffic": COLOUR_TRAFFIC_128 if N == 128 ** 3 else None,
                            "peak_source": src + " hbm_gbs (copy test)"},
            "residual_restrict": {"bound": "hbm", "kernel": "k_restrict_tile<float,4,periodic> (finest)",
                                  "ms_per_launch": ms1, "algorithmic_bytes": bytes1, "achieved": rr_gbs,
                                  "unit": "GB/s", "peak": pk["hbm_gbs"], "frac": rr_gbs / pk["hbm_gbs"],
                                  "traffic": RESTRICT_TRAFFIC_128 if N == 128 ** 3 else None}}


def unet_fwd_flops(n_net):
    """Algorithmic flops of one forward pass of the warm-start U-Net at n_net^3 (3x3x3 convs:
    2 x 27 x Cin x Cout per voxel at the level's resolution; the 1x1 head and glue are ignored)."""
    from paper_2501_13046_gb300 import warmstart as WS
    level = {"e0a": 0, "e0": 0, "e1a": 1, "e1": 1, "e2a": 2, "e2": 2, "ba": 3, "b": 3, "d2a": 2, "d2": 2,
             "d1a": 1, "d1": 1, "d0a": 0, "d0": 0}
    return sum(2 * 27 * cin * cout * (n_net >> level[name]) ** 3 for name, cin, cout in WS.CONVS)


def run_infer(args):
    """Warm-start inference alone (random weights; the cost does not depend on them): the captured
    graph (restriction 128^3 -> 64^3, U-Net, prolongation) replayed per instance."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2501_13046_gb300 import fields
    from paper_2501_13046_gb300 import warmstart as WS
    sc = WS.Scales(s_rho=1e3, s_S=1e6, s_K=1 / 6.0, s_u=0.05, s_W=1e-5)
    pred = WS.Predictor(WS.Params(seed=1), 128, 64, sc)
    pred.capture()
    p = fields.batch_instance(128, 5e-5, 20000, device="cuda")
    u = torch.empty((128,) * 3, dtype=torch.float64, device="cuda")
    W = torch.empty((3,) + (128,) * 3, dtype=torch.float64, device="cuda")
    for _ in range(args.warmup):
        pred.predict_graph(p, u, W)
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ev0.record()
    for _ in range(args.steps):
        pred.predict_graph(p, u, W)
    ev1.record()
    ev1.synchronize()
    ms = ev0.elapsed_time(ev1) / args.steps
    pk, src = peaks()
    tflops = unet_fwd_flops(64) / (ms * 1e-3) / 1e12
    print(json.dumps({"workload": "infer", "ms_per_instance": ms, "instances_per_s": 1e3 / ms,
                      "unet_fwd_gflop": unet_fwd_flops(64) / 1e9, "achieved_tflops": tflops,
                      "bf16_peak_tflops": pk["bf16_tflops"], "frac": tflops / pk["bf16_tflops"],
                      "peak_source": src}))
    return 0


def run_solve_profile(args):
    """Only the benchmarked solve: W + K mixed solves of the 128^3 workload from psi = 1 with the
    settings given (--settings inner,nu,omega; default: autotuned); --workload shell solves the
    256^3 Robin puncture shell instead.  The committed launch lists and kernel captures are taken
    from this command."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2501_13046_gb300 import mg
    if args.workload == "solve":
        p = make_problem()
    elif args.workload == "shell":
        p = fields_mod().puncture_shell(n=args.shell_n)
    else:
        p = fields_mod().bowen_york_binary(n=args.binary_n)
    sp = torch.cuda.current_stream().cuda_stream
    src = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (p["rho0"], p["rho2"], *p["S"])]
    cfg = mg.config_for(p, mg.MG_MIXED, tol=WORKLOAD["tol"], max_outer=60, nested=args.nested)
    if args.settings:
        inner, nu, om = args.settings.split(",")
        apply_tuned(cfg, {"inner_cycles": int(inner), "nu": int(nu), "omega": float(om)})
    else:
        cfg, _ = mg.mg_autotune(cfg, *src, stream=sp)
    ctx = mg.mg_create(cfg, sp)
    mg.mg_set_sources(ctx, *src)
    stream = torch.cuda.current_stream()
    solve_loop(mg, torch, ctx, args.warmup, stream)
    secs, info = solve_loop(mg, torch, ctx, args.steps, stream)
    print(json.dumps({"workload": args.workload, "solves_per_s": args.steps / secs, "outer_iters": info["outer_iters"],
                      "launches_per_solve": info["kernel_launches"], "inner_cycles": cfg.inner_cycles,
                      "nu": cfg.nu_pre, "omega": cfg.omega, "nested": cfg.nested,
                      "nested_iters": info["nested_iters"]}))
    mg.mg_destroy(ctx)
    return 0


def tune_summary(cfg, ms):
    return {"inner_cycles": cfg.inner_cycles, "nu": cfg.nu_pre, "omega": cfg.omega, "tile_waves": cfg.tile_waves,
            "tune_solve_ms": ms}


def apply_tuned(cfg, t):
    cfg.inner_cycles, cfg.nu_pre, cfg.nu_post, cfg.omega = t["inner_cycles"], t["nu"], t["nu"], t["omega"]
    cfg.tile_waves = t.get("tile_waves", 0)
    return cfg


def solve_loop(mg, torch, ctx, steps, stream):
    """steps full solves from psi = 1 on resident sources; returns (seconds via events, last info)."""
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    info = None
    ev0.record(stream)
    for _ in range(steps):
        mg.mg_set_initial_guess(ctx, None, None)
        st, info = mg.mg_solve(ctx)
        assert st == mg.MG_OK, info["history"][-3:]
    ev1.record(stream)
    ev1.synchronize()
    return ev0.elapsed_time(ev1) / 1e3, info


def run_warmstart(args):
    """The learned warm start (its own JSON line): train the U-Net on solver-generated 64^3
    solutions with the library's tcgen05 kernels, then compare warm-started and psi = 1 batched
    mixed-precision solves (and an untrained-network control) on fresh 128^3 instances."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2501_13046_gb300 import fields, mg
    from paper_2501_13046_gb300 import warmstart as WS
    torch.cuda.set_device(0)
    t0 = time.perf_counter()
    data = WS.make_dataset(mg, fields, list(range(10000, 10000 + args.train_samples)), n=64)
    torch.cuda.synchronize()
    t_data = time.perf_counter() - t0
    n_train = len(data)
    sc = WS.fit_scales(data)
    P = WS.Params(seed=1)
    control = WS.Params(seed=1)
    t0 = time.perf_counter()
    hist = WS.train(P, data, sc, epochs=args.epochs, lr=5e-4, warmup=50, minibatch=8)
    torch.cuda.synchronize()
    t_train = time.perf_counter() - t0
    err_train = WS.rel_error(P, sc, data[:16])
    del data
    torch.cuda.empty_cache()
    held = WS.make_dataset(mg, fields, list(range(30000, 30016)), n=64)
    err_held = WS.rel_error(P, sc, held)
    del held
    seeds = list(range(20000, 20000 + args.test_instances))
    out = {}
    for name, PP in (("trained", P), ("untrained_control", control)):
        r = WS.evaluate(mg, fields, PP, sc, seeds, n=128, n_net=64)
        out[name] = {"accepted": int(sum(r["accepted"])), "cold_vcycle_pairs_mean": float(np.mean(r["cold_iters"])),
                     "warm_vcycle_pairs_mean": float(np.mean(r["warm_iters"])), "cold_ms": r["cold_ms"],
                     "warm_ms_incl_inference": r["warm_ms"], "inference_ms": r["infer_ms"],
                     "fallback_ms": r["fallback_ms"], "instances": r["instances"],
                     "dropped_unsolvable": r["dropped_unsolvable"],
                     "cold_solves_per_s": r["instances"] / (r["cold_ms"] * 1e-3),
                     "warm_solves_per_s": r["instances"] / (r["warm_ms"] * 1e-3)}
    line = {"metric": "solves/s to |H|,|M|<=1e-10, learned warm start vs psi=1 (128^3 periodic, batched, mixed)",
            "value": out["trained"]["warm_solves_per_s"], "unit": UNIT, "n_gpus": 1, "higher_is_better": True,
            "dtype": "bf16 network (fp32 accumulate) + f32-inner/f64-outer solver", "data": "synthetic",
            "config": {"workload": "train %d solved 64^3 samples (seeds 10000..), %d epochs; test %d fresh 128^3 "
                                   "instances (seeds 20000..), network run at 64^3 with restriction/prolongation"
                                   % (args.train_samples, args.epochs, args.test_instances),
                       "data_gen_s": t_data, "train_s": t_train, "train_samples_converged": n_train, "loss_first50": float(np.mean(hist[:50])),
                       "loss_last50": float(np.mean(hist[-50:])), "rel_l2_err_train_u_W": err_train,
                       "rel_l2_err_heldout_u_W": err_held, **out}}
    print(json.dumps(line))
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=50)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--workload", default="bench", choices=["bench", "warmstart", "solve", "shell", "binary", "infer"])
    ap.add_argument("--binary-n", type=int, default=128, help="binary workload: cells per axis")
    ap.add_argument("--shell-n", type=int, default=256, help="shell workload: cells per axis")
    ap.add_argument("--settings", default="", help="solve workload: inner_cycles,nu,omega (default: autotune)")
    ap.add_argument("--nested", type=int, default=1, choices=(0, 1),
                    help="nested start of each single-context solve (half-size solve, tricubic start)")
    ap.add_argument("--train-samples", type=int, default=2000)
    ap.add_argument("--epochs", type=int, default=12)
    ap.add_argument("--test-instances", type=int, default=256)
    args = ap.parse_args()
    if args.workload == "warmstart" and args.impl == "ours":
        return run_warmstart(args)
    if args.workload in ("solve", "shell", "binary") and args.impl == "ours":
        return run_solve_profile(args)
    if args.workload == "infer" and args.impl == "ours":
        return run_infer(args)
    if args.impl == "reference":
        return run_reference(args)

    import torch
    ws, rank, local = dist_env()
    torch.cuda.set_device(local)
    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    import __graft_entry__
    if rank == 0:
        __graft_entry__.build()
    if ws > 1:
        dist.barrier()
    __graft_entry__.build()
    from paper_2501_13046_gb300 import mg

    phase("inputs")
    p = make_problem()
    stream = torch.cuda.current_stream()
    sp = stream.cuda_stream
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    src_dev = [dev(a) for a in (p["rho0"], p["rho2"], *p["S"])]

    tuned_params = {}

    def context(precision):
        # one-time launch-parameter tuning (untimed): V-cycles per outer iteration, sweeps, omega
        base = mg.config_for(p, precision, tol=WORKLOAD["tol"], max_outer=60, nested=args.nested)
        cfg, tms = mg.mg_autotune(base, *src_dev, stream=sp)
        tuned_params[precision] = tune_summary(cfg, tms)
        wsz = mg.mg_workspace_size(cfg)
        work = torch.empty(wsz, dtype=torch.uint8, device="cuda")   # torch provides the device memory
        ctx = mg.mg_create(cfg, sp, work)
        mg.mg_set_sources(ctx, *src_dev)
        return ctx, work

    phase("fp64 context and tuning")
    # ---- plain FP64 multigrid (context for the comparison)
    ctx64, w64 = context(mg.MG_FP64)
    solve_loop(mg, torch, ctx64, 1, stream)
    t64, info64 = solve_loop(mg, torch, ctx64, max(1, min(3, args.steps)), stream)
    fp64_solves_per_s = max(1, min(3, args.steps)) / t64
    mg.mg_destroy(ctx64)
    del w64

    phase("mixed context and tuning")
    # ---- the benchmarked path: mixed FP32/FP64
    ctx, work = context(mg.MG_MIXED)
    solve_loop(mg, torch, ctx, args.warmup, stream)
    torch.cuda.synchronize()
    if ws > 1:
        dist.barrier()
    with ClockSampler(local) as clk:
        torch.cuda.synchronize()
        secs, info = solve_loop(mg, torch, ctx, args.steps, stream)
        torch.cuda.synchronize()
    secs = replicas.max_over_ranks(secs, device="cuda")
    value = replicas.job_throughput(args.steps, secs, ws)
    launches = info["kernel_launches"] * args.steps

    phase("timed region done")
    # per-field error of the timed solve (the last one) against the oracle's stored root
    gold = golden("modes_periodic_%d" % WORKLOAD["n"])
    shape = p["rho0"].shape
    u_d = torch.empty(shape, dtype=torch.float64, device="cuda")
    W_d = torch.empty((3,) + shape, dtype=torch.float64, device="cuda")
    mg.mg_get_solution(ctx, u_d, W_d)
    field_err = field_errors(gold, u_d.cpu().numpy(), W_d.cpu().numpy()) if gold else None

    # dominant kernel: one finest-level red-black colour pass (timed live on the context stream)
    roofline = kernel_rooflines(mg, ctx, WORKLOAD["n"] ** 3)

    # the same solve stopped only once every field's last update is <= 1e-10 of its size as well
    cfg_f = mg.config_for(p, mg.MG_MIXED, tol=WORKLOAD["tol"], max_outer=60, nested=args.nested, field_tol=1e-10)
    apply_tuned(cfg_f, tuned_params[mg.MG_MIXED])
    ctx_f = mg.mg_create(cfg_f, sp)
    mg.mg_set_sources(ctx_f, *src_dev)
    solve_loop(mg, torch, ctx_f, 2, stream)
    fsteps = max(1, min(args.steps, 10))
    tf, info_f = solve_loop(mg, torch, ctx_f, fsteps, stream)
    mg.mg_get_solution(ctx_f, u_d, W_d)
    field_acc = {"solves_per_s": fsteps / tf, "outer_iters": info_f["outer_iters"],
                 "nested_outer_iters": info_f["nested_iters"], "final_norms": list(info_f["norms"]),
                 "last_update_rel": list(info_f["rel_change"]),
                 "field_err": field_errors(gold, u_d.cpu().numpy(), W_d.cpu().numpy()) if gold else None,
                 "stop": "max(|H|,|M_i|) <= 1e-10 and every field's last update <= 1e-10 of its max-norm"}
    mg.mg_destroy(ctx_f)
    # ... and with each field's remaining error estimated from its last two updates (field_est)
    cfg_e = mg.config_for(p, mg.MG_MIXED, tol=WORKLOAD["tol"], max_outer=60, nested=args.nested, field_tol=1e-10,
                          field_est=1)
    apply_tuned(cfg_e, tuned_params[mg.MG_MIXED])
    ctx_e = mg.mg_create(cfg_e, sp)
    mg.mg_set_sources(ctx_e, *src_dev)
    solve_loop(mg, torch, ctx_e, 2, stream)
    te, info_e = solve_loop(mg, torch, ctx_e, fsteps, stream)
    mg.mg_get_solution(ctx_e, u_d, W_d)
    field_est = {"solves_per_s": fsteps / te, "outer_iters": info_e["outer_iters"],
                 "nested_outer_iters": info_e["nested_iters"], "final_norms": list(info_e["norms"]),
                 "last_update_rel": list(info_e["rel_change"]),
                 "field_err": field_errors(gold, u_d.cpu().numpy(), W_d.cpu().numpy()) if gold else None,
                 "stop": "max(|H|,|M_i|) <= 1e-10 and every field's estimated remaining error (last update x "
                         "rho / (1 - rho), rho the ratio of its last two updates) <= 1e-10 of its max-norm"}
    mg.mg_destroy(ctx_e)
    del u_d, W_d

    # ---- end to end through the public API with host buffers
    host_src = [torch.from_numpy(np.ascontiguousarray(a)).pin_memory() for a in (p["rho0"], p["rho2"], *p["S"])]
    u_h = torch.empty(shape, dtype=torch.float64).pin_memory()
    W_h = torch.empty((3,) + shape, dtype=torch.float64).pin_memory()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e2e_steps = max(1, min(args.steps, 5))
    ev0.record(stream)
    for _ in range(e2e_steps):
        mg.mg_set_sources(ctx, *[t.numpy() for t in host_src])
        mg.mg_set_initial_guess(ctx, None, None)
        st, _ = mg.mg_solve(ctx)
        mg.mg_get_solution(ctx, u_h.numpy(), W_h.numpy())
    ev1.record(stream)
    ev1.synchronize()
    e2e_secs = ev0.elapsed_time(ev1) / 1e3
    N = int(np.prod(shape))
    e2e = {"value": ws * e2e_steps / e2e_secs, "unit": UNIT, "h2d_bytes_per_step": 5 * N * 8,
           "d2h_bytes_per_step": 4 * N * 8}
    mg.mg_destroy(ctx)
    del work
    torch.cuda.empty_cache()
    phase("shell")
    shell = {}
    q = fields_mod().puncture_shell(n=256)
    qsrc = [dev(a) for a in (q["rho0"], q["rho2"], *q["S"])]
    for name, prec in (("mixed", mg.MG_MIXED), ("fp64_plain", mg.MG_FP64)):
        # the 128^3 periodic tuning of the same precision (a 256^3 FP64 tuning would take minutes);
        # the default settings if that does not converge here
        for params in (tuned_params[prec], None):
            cfgq = mg.config_for(q, prec, tol=WORKLOAD["tol"], max_outer=60, nested=args.nested)
            if params:
                apply_tuned(cfgq, params)
            cq = mg.mg_create(cfgq, sp)
            mg.mg_set_sources(cq, *qsrc)
            try:
                solve_loop(mg, torch, cq, 1, stream)
                tq, iq = solve_loop(mg, torch, cq, 2, stream)
            except (mg.MGError, AssertionError):
                mg.mg_destroy(cq)
                continue
            shell[name] = {"solves_per_s": 2 / tq, "outer_iters": iq["outer_iters"],
                           "max_norm": float(iq["norms"].max()), "settings": "tuned" if params else "default"}
            gq = golden("puncture_shell_256")
            if gq:   # per-field error of the timed solve against the oracle's 256^3 root
                uq = torch.empty(q["rho0"].shape, dtype=torch.float64, device="cuda")
                Wq = torch.empty((3,) + q["rho0"].shape, dtype=torch.float64, device="cuda")
                mg.mg_get_solution(cq, uq, Wq)
                shell[name]["field_err"] = field_errors(gq, uq.cpu().numpy(), Wq.cpu().numpy(),
                                                        psi_background_at(gq, q["punctures"]))
                del uq, Wq
            mg.mg_destroy(cq)
            break
    # the same problem on its octant (128^3, three symmetry planes), mixed
    qo = fields_mod().octant(q)
    qosrc = [dev(a) for a in (qo["rho0"], qo["rho2"], *qo["S"])]
    for params in (tuned_params[mg.MG_MIXED], None):
        cfgo = mg.config_for(qo, mg.MG_MIXED, tol=WORKLOAD["tol"], max_outer=60, nested=args.nested)
        if params:
            apply_tuned(cfgo, params)
        co = mg.mg_create(cfgo, sp)
        mg.mg_set_sources(co, *qosrc)
        try:
            solve_loop(mg, torch, co, 2, stream)
            to, io = solve_loop(mg, torch, co, 5, stream)
        except (mg.MGError, AssertionError):
            mg.mg_destroy(co)
            continue
        shell["mixed_octant_128"] = {"solves_per_s": 5 / to, "outer_iters": io["outer_iters"],
                                     "max_norm": float(io["norms"].max()),
                                     "settings": "tuned" if params else "default",
                                     "workload": "the octant [0,64]^3 at 128^3, symmetry planes x,y,z=0 (reflect=7)"}
        mg.mg_destroy(co)
        break
    del qosrc
    del qsrc
    torch.cuda.empty_cache()
    phase("binary")
    # Bowen-York binary (two boosted, spinning punctures and a scalar shell), 128^3, nested start
    bq = fields_mod().bowen_york_binary(n=128)
    bsrc = [dev(a) for a in (bq["rho0"], bq["rho2"], *bq["S"])]
    binary = {}
    for params in (tuned_params[mg.MG_MIXED], None):
        cfgb = mg.config_for(bq, mg.MG_MIXED, tol=WORKLOAD["tol"], max_outer=60, nested=args.nested)
        if params:
            apply_tuned(cfgb, params)
        cb = mg.mg_create(cfgb, sp)
        mg.mg_set_sources(cb, *bsrc)
        try:
            solve_loop(mg, torch, cb, 2, stream)
            tb, ib = solve_loop(mg, torch, cb, 5, stream)
        except (mg.MGError, AssertionError):
            mg.mg_destroy(cb)
            continue
        binary = {"solves_per_s": 5 / tb, "outer_iters": ib["outer_iters"], "nested_outer_iters": ib["nested_iters"],
                  "max_norm": float(ib["norms"].max()), "settings": "tuned" if params else "default"}
        mg.mg_destroy(cb)
        break
    del bsrc
    torch.cuda.empty_cache()
    phase("sine 32")
    # the 32^3 sine workload (2nd order, L = 16, 4 levels): both precisions
    c1 = fields_mod().sine_periodic(n=32)
    c1src = [dev(a) for a in (c1["rho0"], c1["rho2"], *c1["S"])]
    sine32 = {"workload": "phi = 0.1 sin(2 pi x/L), Pi = 0.05 sin(2 pi y/L), L=16, 32^3, 2nd order, 4 levels, "
                          "K from integrability, psi = 1 start"}
    for name, prec in (("mixed", mg.MG_MIXED), ("fp64_plain", mg.MG_FP64)):
        cx = mg.mg_create(mg.config_for(c1, prec, tol=WORKLOAD["tol"], max_outer=60), sp)
        mg.mg_set_sources(cx, *c1src)
        solve_loop(mg, torch, cx, 3, stream)
        t1, i1 = solve_loop(mg, torch, cx, 20, stream)
        sine32[name] = {"solves_per_s": 20 / t1, "outer_iters": i1["outer_iters"], "max_norm": float(i1["norms"].max())}
        mg.mg_destroy(cx)
    del c1src
    phase("batch mixed")
    batch_mixed = batch_measure(mg, torch, sp, mg.MG_MIXED, repeats=2)
    torch.cuda.empty_cache()
    phase("batch fp64")
    batch_fp64 = batch_measure(mg, torch, sp, mg.MG_FP64, repeats=1)
    torch.cuda.empty_cache()

    if ws > 1:
        dist.barrier()
        dist.destroy_process_group()
    if rank != 0:
        return 0
    cpu = None
    if not args.no_cpu_baseline:
        phase("oracle baseline")
        ncpu = os.cpu_count() or 1
        v, det = oracle_full_size(p, ncpu)
        v1, det1 = oracle_full_size(p, 1)
        from oracle import oracle as O
        c1 = fields_mod().sine_periodic(n=32)
        g1 = O.make_grid(c1["n"], c1["lo"], c1["hi"], c1["order"], c1["bc"])
        sine_cpu = {}
        for th in (ncpu, 1):
            O.set_threads(th)
            t0 = time.perf_counter()
            r1 = O.solve(g1, c1["rho0"], c1["rho2"], c1["S"], O.K_INTEGRABILITY, tol=WORKLOAD["tol"], max_outer=60)
            sine_cpu["threads_%d" % th] = {"solves_per_s": 1.0 / (time.perf_counter() - t0), "outer_iters": r1["iters"]}
        sine32["oracle"] = sine_cpu
        cpu = {"value": v, "unit": UNIT, "cores": det["threads"], "kind": "oracle",
               "sample": "the oracle on the 128^3 workload's own inputs: one residual evaluation (%.1f s) and one outer "
                         "iteration (%.1f s) timed, times its %d iterations to 1e-10 (its stored full run to the FP64 "
                         "floor, tests/golden) = %.0f s per solve"
                         % (det["t_residual_s"], det["t_iteration_s"], det["iters_to_tol"], det["solve_s"]),
               "single_thread": {"value": v1, "solve_s": det1["solve_s"], "t_iteration_s": det1["t_iteration_s"]},
               "cpu_model": cpu_model(),
               "note": "the oracle's Gauss-Seidel sweeps are sequential; only its pointwise loops use OpenMP"}
    cfgd = dict(WORKLOAD, gridpoints_per_s=value * WORKLOAD["n"] ** 3,
                outer_iters=info["outer_iters"], final_norms=list(info["norms"]), K=info["K"],
                field_err=field_err, field_err_note="max over 4096+ stored cells of |gpu - oracle| / max|oracle field|, "
                                                    "oracle root to its FP64 floor (tests/golden)",
                field_accurate=field_acc, field_estimated=field_est,
                start="nested: half-size solve, tricubic start" if args.nested else "psi = 1, W = 0",
                nested_outer_iters=info["nested_iters"],
                fp64_plain_solves_per_s=fp64_solves_per_s, fp64_plain_outer_iters=info64["outer_iters"],
                tuned={"mixed": tuned_params[mg.MG_MIXED], "fp64_plain": tuned_params[mg.MG_FP64],
                       "note": "mg_autotune before the timed region (inner V-cycles, sweeps, omega, then the tiled kernels' z chunking)"},
                mixed_over_fp64=value / ws / fp64_solves_per_s,
                puncture_shell_256={**shell, "workload": "M=1 puncture, [-64,64]^3, 256^3, 4th order, Robin 1/r, "
                                                          "phi=0.02 exp(-(r-10)^2/4), Pi=0.01 phi, K=0"},
                sine_32=sine32,
                bowen_york_binary_128={**binary, "workload": "two Bowen-York punctures m=0.5 at (+-3,0,0), P=(0,+-0.2,0), "
                                                             "S=(0,0,0.1), scalar shell A=0.01 at r=8, [-16,16]^3, "
                                                             "128^3, 4th order, Robin, K=0, mixed"},
                batch_64_uneven={"mixed": batch_mixed, "fp64_plain": batch_fp64,
                                 "mixed_over_fp64": batch_mixed["solves_per_s"] / batch_fp64["solves_per_s"],
                                 "workload": "64 periodic instances, n ~ U{48,64,96,128,160}, L=32, 4th order, "
                                             "a0 ~ U[2e-5, 8e-5], one captured graph per round"},
                l2="inputs larger than L2: FP64 state + sources + residual 14 x 16.8 MB = 235 MB > 129 MB",
                parallelism="replicas" if ws > 1 else "single GPU")
    line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": secs / args.steps * 1e3, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f32-inner/f64-outer", "data": "synthetic",
            "config": cfgd, "roofline": roofline, "cpu_baseline": cpu, "e2e": e2e, "gpu_launches": launches,
            "clocks": clk.summary()}
    phase("done")
    print(json.dumps(line))
    return 0


if __name__ == "__main__":
    sys.exit(main())
