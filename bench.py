#!/usr/bin/env python
"""Throughput of the fused SSP-RK3 vielbein-LB + Cahn-Hilliard step on one or more GB300s.

Metric: node-velocity updates per second, NVU/s = 16 * N_theta * N_phi * steps / time (a full
three-stage step counts once), on the 1024 x 2048 FP32 torus coarsening workload (R = 2, r = 1,
tau = 0.6, A = 0.5, kappa = 5e-4, M = 2.5e-3, noise +-0.01), with the HBM roofline of the stage
kernel, an end-to-end figure through the C ABI with host buffers, and the FP64 CPU oracle timed
on a bounded sample as a reported baseline.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

N > 1 (torchrun) runs N independent replicas, one per GPU (weak scaling; the step itself needs
no collective).  Rank 0 prints one JSON line.
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

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

WORKLOAD = "coarsen_torus_1024x2048"
METRIC = "node-velocity updates/s"
UNIT = "NVU/s"
# Algorithmic HBM bytes per node and step: the 17 state arrays (16 populations + phi) are read 5 times
# (stage 1: U^n; stages 2-3: U_in and U^n) and written 3 times over the three Runge-Kutta stages.
BYTES_PER_NODE_STEP = {"f32": 544, "f64": 1088}
# the FP32 path also carries the low word of phi (an 18th array) for precision: 576 B moved per node-step
BYTES_PER_NODE_STEP_MOVED_F32 = 576
PKEYS = ["R", "r", "n_theta", "n_phi", "dt", "tau", "M", "A", "kappa", "geometry", "advection", "ch_mode"]
TRAFFIC_FILE = os.path.join(ROOT, "profiles", "stage_kernel_fp32_uw3_coarsen_1024x2048.md")


def _args():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=2000)
    ap.add_argument("--warmup", type=int, default=20)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-ensemble", action="store_true")
    ap.add_argument("--no-surrogate", action="store_true")
    ap.add_argument("--coarsening", type=int, default=0, metavar="STEPS",
                    help="run only the three 1024x2048 coarsening runs for STEPS steps each and print their L(t)")
    ap.add_argument("--coarsening-every", type=int, default=1000)
    ap.add_argument("--torus-sizes", action="store_true",
                    help="run only the thin-against-reference torus coarsening over six noise seeds (one ensemble)")
    return ap.parse_args()


def _peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            return json.load(fh), "measured"
    except OSError:
        return {"hbm_gbs": 6800.0}, "fallback"


def _traffic_per_launch():
    """DRAM bytes per stage launch from the committed ncu summary, if it was taken on these sources."""
    from paper_1904_10070_gb300 import build
    try:
        txt = open(TRAFFIC_FILE).read()
    except OSError:
        return None
    vals = {}
    for line in txt.splitlines():
        if ":" in line and line.startswith("- "):
            k, v = line[2:].split(":", 1)
            vals[k.strip()] = v.strip().strip("`")
    if vals.get("stage_source_sha256_16") != build.stage_tag():
        return None
    try:
        return float(vals["dram_bytes_per_launch"])
    except (KeyError, ValueError):
        return None


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled every 200 ms while the timed region runs."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.lines = []

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
            time.sleep(0.3)
        except OSError:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append((time.time(), line.strip()))

    def __exit__(self, *exc):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self, t0=None, t1=None):
        """Median SM clock and the throttle reasons seen in the samples taken between t0 and t1
        (host time; the timed region), or in all samples."""
        if not self.lines:
            return None
        sm, smax, reasons = [], 0.0, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ts, ln in self.lines:
            if t0 is not None and not (t0 <= ts <= t1):
                continue
            parts = [x.strip() for x in ln.split(",")]
            if len(parts) < 8:
                continue
            try:
                sm.append(float(parts[1]))
                smax = max(smax, float(parts[2]))
            except ValueError:
                continue
            for nm, val in zip(names, parts[4:8]):
                if val.lower() in ("active", "1", "yes"):
                    reasons.add(nm)
        if not sm:
            return None
        return {"sm_mhz": float(np.median(sm)), "sm_max_mhz": smax, "reasons": sorted(reasons),
                "samples": len(sm), "window": "timed region" if t0 is not None else "whole run"}


def reduce_max(values, dist=None, device="cpu"):
    """Max over ranks of a list of floats (each rank's timings); identity without a process group."""
    if dist is None:
        return list(values)
    import torch
    t = torch.tensor(list(values), dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return [float(x) for x in t]


def aggregate_value(world: int, units_per_rank: float, seconds_max: float) -> float:
    """Whole-job throughput: every rank processed units_per_rank; the job took the slowest rank's time."""
    return world * units_per_rank / seconds_max


def _dist():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def _oracle_sample(rows: int):
    from oracle import vlb_oracle as O
    from paper_1904_10070_gb300 import inputs
    w = inputs.workload(WORKLOAD)
    p = dict(w["params"])
    p["n_theta"] = rows
    geo = O.Geometry(O.Params(**{k: p[k] for k in PKEYS}))
    phi = inputs.noise(1, rows, p["n_phi"], 0.01)
    f, ph = O.init_state(np.ones_like(phi), 0 * phi, 0 * phi, phi)
    return O, geo, f, ph, p["n_phi"]


def _calibrated_rows(target_s: float, steps: int) -> int:
    """theta rows of a 2048-wide sub-grid that the oracle steps `steps` times in about target_s seconds."""
    O, geo, f, ph, ns = _oracle_sample(32)
    t0 = time.perf_counter()
    O.step(f, ph, geo)
    rate = 32 * ns / (time.perf_counter() - t0)  # node-steps per second
    # larger grids run slower per node (memory-bound numpy temporaries): keep a factor 2 of margin
    return int(max(1, min(1024, 0.5 * target_s * rate / (ns * steps))))


def _oracle_worker(args):
    """One host core: the oracle steps its own sub-grid of the workload (a process of the pool)."""
    rows, steps = args
    O, geo, f, ph, ns = _oracle_sample(rows)
    t0 = time.perf_counter()
    O.run(f, ph, geo, steps)
    return time.perf_counter() - t0


def _cpu_model():
    try:
        for line in open("/proc/cpuinfo"):
            if line.lower().startswith(("model name", "cpu part", "hardware")):
                return line.split(":", 1)[1].strip()
    except OSError:
        pass
    import platform
    return platform.processor() or platform.machine()


def cpu_baseline(steps: int = 2, target_s: float = 12.0):
    """The FP64 oracle as it stands, on bounded sub-grids of the workload: once on one core, then on
    every host core at once (one spawned process per core, each stepping its own sub-grid of the same
    size with numpy held to one thread; throughput = all node updates / the slowest process)."""
    import multiprocessing as mp
    rows = _calibrated_rows(target_s, steps)
    ncores = len(os.sched_getaffinity(0)) if hasattr(os, "sched_getaffinity") else (os.cpu_count() or 1)
    ns = 2048
    t1 = _oracle_worker((rows, steps))
    single = 16.0 * rows * ns * steps / t1
    # all cores: 128-row sub-grids (a few hundred MB of numpy temporaries per process), enough steps
    # for about as long as the single-core run
    rows_mc = min(rows, 128)
    steps_mc = max(2, int(round(steps * rows / rows_mc)))
    for var in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS"):
        os.environ[var] = "1"  # inherited by the spawned workers: one thread each
    ctx = mp.get_context("spawn")
    t0 = time.perf_counter()
    with ctx.Pool(ncores) as pool:
        times = pool.map(_oracle_worker, [(rows_mc, steps_mc)] * ncores)
    wall = time.perf_counter() - t0
    allc = 16.0 * rows_mc * ns * steps_mc * ncores / max(times)
    return {"value": allc, "unit": UNIT, "cores": ncores, "kind": "oracle",
            "single_core_value": single, "cpu_model": _cpu_model(), "nproc": os.cpu_count(),
            "sample": f"FP64 numpy oracle on sub-grids of the workload (same parameters): one core, {steps} "
                      f"SSP-RK3 steps on {rows}x{ns} in {t1:.1f} s; {ncores} cores, one process each stepping "
                      f"its own {rows_mc}x{ns} sub-grid {steps_mc} times, slowest {max(times):.1f} s "
                      f"(pool wall {wall:.1f} s)"}


def run_reference(args):
    """--impl reference: the oracle timed per step on a bounded sample sized for a few minutes in total."""
    rows = _calibrated_rows(120.0, args.steps + args.warmup)
    O, geo, f, ph, ns = _oracle_sample(rows)
    for _ in range(args.warmup):
        f, ph = O.step(f, ph, geo)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        f, ph = O.step(f, ph, geo)
    dt = time.perf_counter() - t0
    val = 16.0 * rows * ns * args.steps / dt
    sample = f"FP64 numpy oracle, {args.steps} steps on a {rows}x{ns} sub-grid of the workload"
    line = {"impl": "reference", "metric": METRIC, "value": val, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * dt / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": {"workload": WORKLOAD, "grid": [rows, ns], "sample": True},
            "cpu_baseline": {"value": val, "unit": UNIT, "cores": 1, "kind": "oracle", "sample": sample},
            "e2e": {"value": val, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def ensemble_measurement(steps: int = 60, seq_steps: int = 10):
    """The 48-tori ensemble: the autotuner's choice, then each execution mode at its best tile height --
    one batched launch per stage (graph-replayed) and one persistent cooperative launch per block of
    steps (grid barrier between stages) -- and the same members stepped one after another with
    per-member launches.  All timed with CUDA events on the ensemble's stream."""
    import torch
    from paper_1904_10070_gb300 import inputs, vlb
    work = inputs.ensemble_workload(48)
    params = []
    for w in work:
        p = dict(w["params"], dt=1.0)
        p["dt"] = 0.5 * vlb.vlb_max_stable_dt(vlb.make_params(**p))
        params.append(vlb.make_params(**p, precision=vlb.FP32))
    ens = vlb.Ensemble(params)
    for v, w in zip(ens.views, work):
        vlb.vlb_set_fields(v, w["rho"], w["ut"], w["up"], w["phi"])
    st = ens.stream
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)

    def timed(n, fn):
        torch.cuda.synchronize()
        e0.record(st)
        fn(n)
        e1.record(st)
        e1.synchronize()
        return e0.elapsed_time(e1) / n

    ens.step(3)  # autotune + graph recording
    chosen = ens.config()
    ms = timed(steps, ens.step)
    per_mode = {}
    for mode, name, rows in ((vlb.ENS_BATCHED, "batched", 16 if chosen["ms"][0] <= chosen["ms"][1] else 8),
                             (vlb.ENS_PERSISTENT, "persistent", 16 if chosen["ms"][2] <= chosen["ms"][3] else 8)):
        ens.configure(mode=mode, tile_rows=rows)
        ens.step(3)
        per_mode[name] = {"tile_rows": rows, "ms_per_step": timed(steps, ens.step)}
    ms_seq = timed(seq_steps, lambda n: [vlb.vlb_step(v, n) for v in ens.views])
    nodes = sum(p.n_theta * p.n_phi for p in params)
    ok = all(np.all(np.isfinite(vlb.vlb_get_totals(v))) for v in ens.views)
    ens.close()
    return {"members": 48, "nodes": nodes, "value": 16.0 * nodes / (ms * 1e-3), "unit": UNIT,
            "ms_per_step": ms, "chosen": {"mode": chosen["mode"], "tile_rows": chosen["tile_rows"]},
            "autotune_ms_stage0": {"batched16": chosen["ms"][0], "batched8": chosen["ms"][1],
                                   "persistent16": chosen["ms"][2], "persistent8": chosen["ms"][3]},
            "modes": per_mode, "sequential_ms_per_step": ms_seq, "speedup_vs_sequential": ms_seq / ms,
            "finite": ok,
            "what": "48 tori, R/r in [1.3, 5], grids 64x128..512x1024, FP32 UW3, per-torus dt; the autotuner's "
                    "choice among batched launches per stage and one persistent cooperative launch (grid barrier "
                    "between stages), 16- or 8-row tiles, vs per-member launches"}


def surrogate_measurement(ntraj: int = 2000, pairs: int = 4, spacing: int = 600, start: int = 300, epochs: int = 3,
                          seeds=(20001, 20002, 20003, 20004), warm: int = 400, nwin: int = 1000, check: int = 3,
                          corr=(4.0, 20.0), judges=("l2", "linf")):
    """The learned surrogate on 256 x 512 tori (R / r in [1.5, 4], seeded quenched noise): trained here on
    `ntraj` solver trajectories by the library's kernels, then advancing each held-out torus by `nwin`
    windows of 50 steps through vlb_surrogate_advance, judged by the solver every `check` windows --
    once with the relative L2 error of phi <= 1e-2 as the judge, once with the relative L-infinity error
    <= 1e-2 -- beside the plain solver from the same state.  Every window is timed with CUDA events on its
    stream; the domain length L_d = A / L_I of both runs is read after every window, outside the timing."""
    import torch
    from paper_1904_10070_gb300 import surrogate as S
    from paper_1904_10070_gb300 import inputs, vlb
    H, W = 256, 512
    t0 = time.perf_counter()
    ds = S.generate(list(range(10000, 10000 + ntraj)), H, W, window=50, pairs=pairs, spacing=spacing, start=start,
                    corr=corr)
    torch.cuda.synchronize()
    gen_s = time.perf_counter() - t0
    tr = S.Trainer(S.SurrogateNet(H, W, seed=1), S.target_ratios(ds), ds.s_n, ds.s_u,
                   weights=(1.0, 0.25, 0.25, 0.25))
    n_pairs = len(ds)
    _, train_s = tr.fit(ds, epochs=epochs, lr=1e-3)
    del ds
    torch.cuda.empty_cache()

    def run(norm, floor):
        t_ref = t_sur = 0.0
        ld_dev, ld_curves, errs, errs_inf, kinds_all = [], [], [], [], []
        ld_ref_all, ld_sur_all, ld_twin_all = [], [], []
        for seed in seeds:
            R = S.radius_for(seed)
            p = S.member_params(R, H, W)
            phi = S.initial_phi(seed, H, W)
            z = np.zeros_like(phi)

            def solver(dphi=None):
                s = vlb.Solver(vlb.make_params(**p, precision=vlb.FP32), stream=torch.cuda.Stream())
                s.set_fields(np.ones_like(phi), z, z, phi if dphi is None else phi + dphi)
                s.step(warm)
                return s

            ref, sur = solver(), solver()
            # the noise floor of a single trajectory's L_d: the solver from phi + 1e-6 noise
            twin = solver(1e-6 * inputs.noise(seed + 7, H, W, 1.0)) if floor else None
            adv = S.Advancer(tr, sur, window=50, check_every=check, phi_tol=1e-2, norm=norm)
            area = 4.0 * math.pi ** 2 * p["r"] * p["R"]
            curve = []
            for k in range(nwin):
                for s_, fn in ((ref, lambda: ref.step(50)), (sur, lambda: adv.advance(1))):
                    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                    torch.cuda.synchronize()
                    e0.record(s_.stream)
                    fn()
                    e1.record(s_.stream)
                    e1.synchronize()
                    if s_ is ref:
                        t_ref += e0.elapsed_time(e1)
                    else:
                        t_sur += e0.elapsed_time(e1)
                if twin is not None:
                    twin.step(50)
                    ld_twin_all.append(area / twin.interface_length())
                l_ref, l_sur = area / ref.interface_length(), area / sur.interface_length()
                ld_dev.append(abs(l_sur / l_ref - 1.0))
                ld_ref_all.append(l_ref)
                ld_sur_all.append(l_sur)
                if k % 50 == 49:
                    curve.append([50 * (k + 1), round(l_ref, 5), round(l_sur, 5)])
            ld_curves.append({"R": round(R, 4), "t_steps_Ld_solver_Ld_surrogate": curve})
            errs += adv.errors
            errs_inf += adv.errors_linf
            kinds_all += adv.kinds
            adv.close()
            ref.close()
            sur.close()
            if twin is not None:
                twin.close()
        n = len(seeds) * nwin
        # a prediction that overflowed has a non-finite error: the judge rejected it (a fallback)
        fin = [float(e) for e in errs if math.isfinite(e)]
        fin_inf = [float(e) for e in errs_inf if math.isfinite(e)]
        # the coarsening curve: L_d averaged over the held-out tori, window by window
        mean_ref = np.mean(np.reshape(ld_ref_all, (len(seeds), nwin)), axis=0)
        mean_sur = np.mean(np.reshape(ld_sur_all, (len(seeds), nwin)), axis=0)
        floor_out = None
        if ld_twin_all:
            twin_dev = np.abs(np.array(ld_twin_all) / np.array(ld_ref_all) - 1.0)
            mean_twin = np.mean(np.reshape(ld_twin_all, (len(seeds), nwin)), axis=0)
            floor_out = {"what": "the solver against itself from phi + 1e-6 noise: the chaotic spread of one "
                                 "trajectory's L_d over the same horizon",
                         "Ld_max_rel_dev": float(np.max(twin_dev)),
                         "Ld_rel_dev_final_mean": float(np.mean(twin_dev[nwin - 1::nwin])),
                         "mean_curve_max_rel_dev": float(np.max(np.abs(mean_twin / mean_ref - 1.0)))}
        judged = kinds_all.count("checked") + kinds_all.count("fallback")
        return {"judge": f"relative {'L2' if norm == 'l2' else 'L-infinity'} error of phi <= 1e-2 on every "
                         f"{check}th window (solver result kept)",
                "windows": n, "predicted_windows": kinds_all.count("surrogate"),
                "fallbacks": kinds_all.count("fallback"), "fallback_rate_of_judged": kinds_all.count("fallback") / max(judged, 1),
                "solver_ms_per_window": t_ref / n, "surrogate_ms_per_window": t_sur / n, "speedup": t_ref / t_sur,
                "phi_l2_err_max": max(fin) if fin else None, "phi_l2_err_median": float(np.median(fin)) if fin else None,
                "phi_linf_err_max": max(fin_inf) if fin_inf else None,
                "nonfinite_predictions": len(errs) - len(fin),
                "Ld_max_rel_dev": max(ld_dev), "Ld_rel_dev_final_mean": float(np.mean(ld_dev[nwin - 1::nwin])),
                "mean_curve_max_rel_dev": float(np.max(np.abs(mean_sur / mean_ref - 1.0))),
                "mean_curve_final_rel_dev": float(mean_sur[-1] / mean_ref[-1] - 1.0),
                "noise_floor": floor_out, "Ld_curves_every_50_windows": ld_curves}

    out = {"workload": "surrogate_torus_256x512 (R/r in [1.5, 4], quenched seeded noise, FP32 solver)",
           "train_trajectories": ntraj, "train_pairs": n_pairs, "train_iters": n_pairs * epochs,
           "gen_s": gen_s, "train_s": train_s, "window_steps": 50, "check_every": check,
           "held_out_tori": len(seeds), "windows_per_torus": nwin, "warm_start_steps": warm}
    out["train_domain_scale_cells"] = list(corr) if corr else S.CORR_CELLS
    for k, j in enumerate(judges):
        out[f"{j}_judge"] = run(j, floor=k == 0)
    # headline figures: the L2 judge
    for k in ("speedup", "fallbacks", "Ld_max_rel_dev", "mean_curve_max_rel_dev", "phi_l2_err_max", "phi_linf_err_max",
              "solver_ms_per_window", "surrogate_ms_per_window"):
        out[k] = out["l2_judge"][k]
    return out


def stabilised_measurement(steps: int = 200):
    """The coarsening workload with the stabilised semi-implicit Cahn-Hilliard stages (ch_stab = 1):
    ms per step at its own stable step, and simulated time per wall second against the explicit step
    at the explicit limit (CUDA events on the solver's stream, FP32, same initial state)."""
    import torch
    from paper_1904_10070_gb300 import inputs, vlb
    w = inputs.workload(WORKLOAD)
    out = {}
    for stab in (0, 1):
        p = dict(w["params"])
        dt_max = vlb.vlb_max_stable_dt(vlb.make_params(**{k: p[k] for k in PKEYS}, ch_stab=stab))
        p["dt"] = min(p["dt"], dt_max) if stab == 0 else 0.8 * dt_max
        s = vlb.Solver(vlb.make_params(**{k: p[k] for k in PKEYS}, precision=vlb.FP32, ch_stab=stab))
        s.set_fields(w["rho"], w["ut"], w["up"], w["phi"])
        s.step(5)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        e0.record(s.stream)
        s.step(steps)
        e1.record(s.stream)
        e1.synchronize()
        ms = e0.elapsed_time(e1) / steps
        finite = bool(np.all(np.isfinite(s.totals())))
        s.close()
        out["stabilised" if stab else "explicit"] = {"dt": p["dt"], "ms_per_step": ms,
                                                      "simulated_time_per_s": p["dt"] / (ms * 1e-3), "finite": finite}
    out["speedup_simulated_time"] = (out["stabilised"]["simulated_time_per_s"] /
                                     out["explicit"]["simulated_time_per_s"])
    out["what"] = ("1024x2048 coarsening workload: explicit step at the workload dt (its Cahn-Hilliard limit) vs "
                   "the stabilised semi-implicit Cahn-Hilliard stages at 0.8 of their own stable dt")
    return out


def coarsening_runs(steps: int = 50000, every: int = 1000, dt_cap: float = 5e-4):
    """Spinodal coarsening from noise +-0.01 on the 1024 x 2048 grid (R = 2, r = 1; A = 0.5,
    kappa = 5e-4, M = 2.5e-3; Sec. 4.1): the hydrodynamic run (tau = 0.6), the diffusive run (no
    advection in Eq. CH and no force on the fluid, tau = 6) and the flat periodic control
    (2 pi r x 2 pi R, square cells), FP32 with the stabilised Cahn-Hilliard stages at
    dt = min(the paper's 5e-4, 0.8 of their stable dt).  Every `every` steps: the domain length
    L_d = A_total / L_I (Eq. cart_scaling_L0) and the structure-factor length L_S, the phi total
    (conserved) and max |u|.  The growth exponent is the least-squares slope of log L against log t
    over the second half of the samples."""
    import torch
    from paper_1904_10070_gb300 import inputs, vlb
    runs = {"hydro_torus": dict(geometry=0, ch_mode=0, tau=0.6),
            "diffusive_torus": dict(geometry=0, ch_mode=1, tau=6.0),
            "hydro_flat": dict(geometry=1, ch_mode=0, tau=0.6)}
    out = {"steps": steps, "every": every}
    for name, over in runs.items():
        w = inputs.workload("coarsen_torus_1024x2048")
        p = dict(w["params"], **over)
        dt_max = vlb.vlb_max_stable_dt(vlb.make_params(**{k: p[k] for k in PKEYS}, ch_stab=1))
        p["dt"] = min(dt_cap, 0.8 * dt_max)
        s = vlb.Solver(vlb.make_params(**{k: p[k] for k in PKEYS}, precision=vlb.FP32, ch_stab=1))
        s.set_fields(w["rho"], w["ut"], w["up"], w["phi"])
        area = 4.0 * math.pi ** 2 * p["r"] * p["R"]
        tot0 = s.totals()
        rec = {"t": [], "L_d": [], "L_S": [], "max_u": []}
        ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        step_ms = 0.0
        for k in range(steps // every):
            ev0.record(s.stream)
            s.step(every)
            ev1.record(s.stream)
            ev1.synchronize()
            step_ms += ev0.elapsed_time(ev1)
            L_I = s.interface_length()
            rec["t"].append((k + 1) * every * p["dt"])
            rec["L_d"].append(area / L_I if L_I > 0 else math.inf)
            rec["L_S"].append(s.structure_length())
            rec["max_u"].append(float(s.totals()[3]))
        tot1 = s.totals()
        s.close()

        def slope(key):
            t, L = np.array(rec["t"]), np.array(rec[key])
            h = len(t) // 2
            ok = np.isfinite(L[h:]) & (L[h:] > 0)
            if ok.sum() < 2:
                return None
            return float(np.polyfit(np.log(t[h:][ok]), np.log(L[h:][ok]), 1)[0])

        out[name] = dict(dt=p["dt"], tau=p["tau"], ch_mode=p["ch_mode"], geometry=p["geometry"],
                         ms_per_step=step_ms / (steps // every * every), finite=bool(np.all(np.isfinite(tot1))),
                         phi_total_drift=float(abs(tot1[1] - tot0[1]) / max(abs(tot0[1]), 1e-30)),
                         phi_total=[float(tot0[1]), float(tot1[1])],
                         exponent_L_d=slope("L_d"), exponent_L_S=slope("L_S"), **rec)
    return out


def torus_size_seeds(seeds=(6, 7, 8, 9, 10, 11), t_marks=(10, 30, 50, 70, 100, 140, 170, 200, 225, 250)):
    """Thin against reference torus (Sec. 4.1.2): even-mixture coarsening from noise +-0.1 at n0 = 20 on
    R = 2.5, r = 1 and R = 5, r = 0.5, 400 x 800, one ensemble member per (torus, seed) in one launch per
    stage at a common dt (0.9 of the smaller stable step, at most 5e-4).  L_d = A / L_I at each mark; the
    apparent exponent over t >= 140 per member, its mean and spread per torus, and the exponent of the
    seed-averaged curve."""
    from paper_1904_10070_gb300 import inputs, vlb
    tori = (("reference", 2.5, 1.0), ("thin", 5.0, 0.5))

    def pd(R, r):
        return dict(geometry=0, R=R, r=r, n_theta=400, n_phi=800, dt=1.0, tau=2.5e-3, M=2.5e-3, A=0.5, kappa=5e-4,
                    advection=0, ch_mode=0)

    dt = min([5e-4] + [0.9 * vlb.vlb_max_stable_dt(vlb.make_params(**pd(R, r))) for _, R, r in tori])
    mem = [(name, R, r, seed) for seed in seeds for name, R, r in tori]
    ens = vlb.Ensemble([vlb.make_params(**dict(pd(R, r), dt=dt), precision=vlb.FP32) for _, R, r, _ in mem])
    for v, (_, _, _, seed) in zip(ens.views, mem):
        phi = inputs.noise(seed, 400, 800, 0.1)
        z = np.zeros_like(phi)
        vlb.vlb_set_fields(v, np.full_like(phi, 20.0), z, z, phi)
    done, Ld = 0, [[] for _ in mem]
    t0 = time.perf_counter()
    for t in t_marks:
        n = int(round(t / dt)) - done
        ens.step(n)
        done += n
        for k, (v, (_, R, r, _)) in enumerate(zip(ens.views, mem)):
            Ld[k].append(4 * math.pi ** 2 * R * r / vlb.vlb_interface_length(v))
    wall = time.perf_counter() - t0
    ens.close()
    t = np.array(t_marks, float)
    late = t >= 140
    out = {"dt": dt, "steps": done, "wall_s": wall, "t": list(t_marks), "members": []}
    for k, (name, _, _, seed) in enumerate(mem):
        e = float(np.polyfit(np.log(t[late]), np.log(np.array(Ld[k])[late]), 1)[0])
        out["members"].append({"torus": name, "seed": seed, "exponent_late": e, "L_d": [round(x, 4) for x in Ld[k]]})
    for name, _, _ in tori:
        es = [m["exponent_late"] for m in out["members"] if m["torus"] == name]
        curve = np.mean([Ld[k] for k, m in enumerate(mem) if m[0] == name], axis=0)
        out[name] = {"exponent_mean": float(np.mean(es)), "exponent_spread": float(np.std(es)),
                     "exponent_of_mean_curve": float(np.polyfit(np.log(t[late]), np.log(curve[late]), 1)[0]),
                     "mean_L_d": [round(float(x), 4) for x in curve]}
    return out


def main():
    args = _args()
    world, rank, local = _dist()
    if args.impl == "reference":
        if rank == 0:
            run_reference(args)
        return
    import torch
    from paper_1904_10070_gb300 import inputs, vlb

    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA GPU")
    torch.cuda.set_device(local)
    if args.coarsening > 0:
        if rank == 0:
            print(json.dumps({"coarsening": coarsening_runs(args.coarsening, args.coarsening_every)}), flush=True)
        return
    if args.torus_sizes:
        if rank == 0:
            print(json.dumps({"torus_sizes": torus_size_seeds()}), flush=True)
        return
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))

    def barrier():
        if dist is not None:
            dist.barrier()

    w = inputs.workload(WORKLOAD)
    p = w["params"]
    N = p["n_theta"] * p["n_phi"]
    params = vlb.make_params(**{k: p[k] for k in PKEYS}, precision=vlb.FP32)
    solver = vlb.Solver(params)
    stream = solver.stream
    solver.set_fields(w["rho"], w["ut"], w["up"], w["phi"])
    for _ in range(args.warmup):
        vlb.vlb_step(solver.h, 1)
    torch.cuda.synchronize()
    barrier()

    # Timed region: blocks of exactly K steps, each bracketed by a barrier and a synchronize and timed
    # with CUDA events on the solver's stream; enough blocks to fill about a second, so that the clock
    # samples (every 200 ms) fall inside it.  ms = the median block.
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ev0.record(stream)
    vlb.vlb_step(solver.h, args.steps)
    ev1.record(stream)
    ev1.synchronize()
    est_s = max(ev0.elapsed_time(ev1) * 1e-3, 1e-6)
    nblocks = int(min(500, max(5, np.ceil(1.0 / est_s))))
    nblocks = int(reduce_max([nblocks], dist, device="cuda")[0])
    block_ms = []
    with ClockSampler(local) as clk:
        t_on = time.time()
        for _ in range(nblocks):
            torch.cuda.synchronize()
            barrier()
            ev0.record(stream)
            vlb.vlb_step(solver.h, args.steps)
            ev1.record(stream)
            ev1.synchronize()
            torch.cuda.synchronize()
            barrier()
            block_ms.append(ev0.elapsed_time(ev1))
        t_off = time.time()
        time.sleep(0.25)  # let the sampler deliver the last in-window sample
    block_ms = reduce_max(block_ms, dist, device="cuda")  # max over ranks, block by block
    ms = float(np.median(block_ms))
    clocks = clk.summary(t_on, t_off) or clk.summary()
    tot = solver.totals()
    if not np.all(np.isfinite(tot)):
        raise SystemExit(f"non-finite totals after the timed steps: {tot}")

    # end to end through the C ABI with pinned host buffers: set fields -> K steps -> read fields
    pin = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).pin_memory().numpy()  # noqa: E731
    h_in = [pin(w["rho"]), pin(w["ut"]), pin(w["up"]), pin(w["phi"])]
    h_out = [pin(np.empty((p["n_theta"], p["n_phi"]))) for _ in range(5)]
    torch.cuda.synchronize()
    barrier()
    t0 = time.perf_counter()
    vlb.vlb_set_fields(solver.h, *h_in)
    vlb.vlb_step(solver.h, args.steps)
    vlb.vlb_get_fields(solver.h, p["n_theta"], p["n_phi"], out=h_out)
    e2e_s = time.perf_counter() - t0
    barrier()

    ms, e2e_s = reduce_max([ms, e2e_s], dist, device="cuda")
    solver.close()
    if rank != 0:
        if dist is not None:
            dist.destroy_process_group()
        return

    value = aggregate_value(world, 16.0 * N * args.steps, ms * 1e-3)
    peaks, peak_kind = _peaks()
    step_s = ms * 1e-3 / args.steps
    launch_s = step_s / 3.0  # every launch of the step is the stage kernel
    alg_bytes_launch = BYTES_PER_NODE_STEP["f32"] * N / 3.0
    achieved = alg_bytes_launch / launch_s / 1e9
    moved = BYTES_PER_NODE_STEP_MOVED_F32 * N / 3.0 / launch_s / 1e9
    traffic = _traffic_per_launch()
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": WORKLOAD, "grid": [p["n_theta"], p["n_phi"]], "R": p["R"], "r": p["r"],
                   "precision": "fp32 state, fp64 coefficients and sums", "advection": "uw3",
                   "ch_mode": "hydrodynamic", "parallelism": f"replicas x{world}",
                   "l2": "no flush: one step moves 576 B x 2.1 M nodes = 1.2 GB through a 126 MB L2",
                   "timed_blocks": {"blocks": nblocks, "steps_each": args.steps, "ms_median": ms,
                                    "ms_min": float(np.min(block_ms)), "ms_max": float(np.max(block_ms))}},
        "roofline": {"bound": "hbm", "achieved": achieved, "peak": peaks["hbm_gbs"], "unit": "GB/s",
                     "frac": achieved / peaks["hbm_gbs"], "traffic": traffic,
                     "kernel": "stage_kernel<float,UW3,HYDRO>",
                     "peak_source": f"{peak_kind} hbm_gbs (copy)",
                     "algorithmic_bytes_per_launch": alg_bytes_launch,
                     "algorithmic_bytes": "544 B per node-step: 17 arrays x (5 reads + 3 writes) x 4 B",
                     "moved_with_phi_lo": {"bytes_per_node_step": BYTES_PER_NODE_STEP_MOVED_F32,
                                           "achieved": moved, "frac": moved / peaks["hbm_gbs"]}},
        "e2e": {"value": aggregate_value(world, 16.0 * N * args.steps, e2e_s), "unit": UNIT,
                "h2d_bytes_per_step": 4 * N * 8 / args.steps, "d2h_bytes_per_step": 5 * N * 8 / args.steps,
                "what": "vlb_set_fields (host) + vlb_step(K) + vlb_get_fields (host), wall clock"},
        "gpu_launches": 3 * args.steps,  # per timed block of K steps
        "clocks": clocks,
    }
    if world == 1 and not args.no_ensemble:
        line["ensemble"] = ensemble_measurement()
    if world == 1:
        line["stabilised_ch"] = stabilised_measurement()
    if world == 1 and not args.no_surrogate:
        line["surrogate"] = surrogate_measurement()
    if world == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline()
    print(json.dumps(line), flush=True)
    if dist is not None:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
