"""Benchmark of the ionization step on GB300.

Workload (default): nitrogen, 256x256x512 = 33,554,432 cells, one step of
dt = 0.05 fs per timed iteration, FP32 populations with FP64 Bateman
coefficients for nearly degenerate cells (ion_step, ION_F32).  Each timed
iteration restores the pristine input state (untimed), flushes L2 (untimed),
then times one ion_step with CUDA events on the launching stream.

Printed: one JSON line with the metric (cell-updates/s), the roofline of the
dominant kernel, the plain FP64 form on the same inputs, the end-to-end
number through host buffers, the FP64 CPU oracle on a bounded sample, and
the SM clocks sampled during the timed region.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

With --gpus N > 1 (under torchrun) every rank runs its own full-size shard
(weak scaling, no data-path collective); rank 0 prints.
"""
from __future__ import annotations

import argparse
import json
import os
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "cell-updates/s"
WORKLOAD = "nitrogen_3d_256x256x512_fp32_fp64fallback"
GRID = (256, 256, 512)
FALLBACK_HBM_GBS = 6800.0


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=300)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--e2e-chunks", type=int, default=16,
                    help="cell chunks of the pipelined end-to-end run")
    ap.add_argument("--no-batched", action="store_true")
    ap.add_argument("--no-krypton", action="store_true")
    ap.add_argument("--no-surrogate", action="store_true")
    return ap.parse_args()


TRAFFIC_FILE = os.path.join(ROOT, "profiles", "traffic_nitrogen_3d.txt")
ISSUE_FILE = os.path.join(ROOT, "profiles", "issue_batched_mixed.txt")
KERNEL_SOURCES = ["paper_2202_10647_gb300/csrc/step_f32.cu",
                  "paper_2202_10647_gb300/csrc/ion_device.cuh",
                  "paper_2202_10647_gb300/csrc/ion_cell.cuh",
                  "paper_2202_10647_gb300/csrc/ion_step.cuh"]


def kernel_sources_hash() -> str:
    """sha256 over the sources of the step's three FP32 kernels."""
    import hashlib
    h = hashlib.sha256()
    for rel in KERNEL_SOURCES:
        with open(os.path.join(ROOT, rel), "rb") as f:
            h.update(f.read())
    return h.hexdigest()


def _recorded(path):
    """key: value lines of a committed ncu record, or None when the record
    was taken on other kernel sources."""
    if not os.path.exists(path):
        return None
    kv = {}
    with open(path) as f:
        for line in f:
            if ":" in line and not line.startswith("#"):
                k, v = line.split(":", 1)
                kv[k.strip()] = v.strip()
    if kv.get("sources_sha256") != kernel_sources_hash():
        return None
    return kv


def recorded_issue_shape():
    """The launch shape (cells per lane, warps per block, blocks per SM) the
    committed instruction counts of the batched step were captured with."""
    kv = _recorded(ISSUE_FILE)
    try:
        return tuple(int(x) for x in kv["shape"].split(","))
    except (TypeError, KeyError, ValueError):
        return None


def batched_issue_roofline(ms, sm_mhz, num_sms):
    """Issue roofline of the batched step: the warp instructions of one step
    (committed ncu record, in the launch shape it was captured with; `ms` is
    the step's time in that shape) against 4 warp instructions per SM cycle
    at the SM clock sampled during the run, and each kernel's share."""
    kv = _recorded(ISSUE_FILE)
    if kv is None or not sm_mhz:
        return None
    try:
        inst = float(kv["warp_inst_per_step"])
        per = {k: (float(kv[f"{k}_warp_inst"]), float(kv[f"{k}_us"]))
               for k in ("stream", "stiff", "fb")}
        scale = float(kv["scale"])
    except (KeyError, ValueError):
        return None
    peak = num_sms * 4 * sm_mhz * 1e6  # warp instructions per second
    achieved = inst / (ms * 1e-3)
    kernels = {}
    for k, (ki, kus) in per.items():
        # in the capture: the kernel's own issue rate against the ceiling
        kernels[f"ion_{k}_kernel"] = {
            "warp_inst_per_step": ki * scale,
            "issue_frac_in_capture": ki / (kus * 1e-6) / peak if kus > 0 else None}
    return {"bound": "issue", "achieved": achieved / 1e9, "peak": peak / 1e9,
            "unit": "G warp instructions/s", "frac": achieved / peak,
            "warp_inst_per_step": inst, "kernels": kernels, "ms_per_step": ms,
            "launch_shape": list(recorded_issue_shape() or ()),
            "record": os.path.relpath(ISSUE_FILE, ROOT)}


def recorded_traffic():
    """DRAM bytes of one full-size step from the committed ncu summary, or
    None when the summary was taken on other kernel sources."""
    kv = _recorded(TRAFFIC_FILE)
    try:
        return None if kv is None else int(kv["dram_bytes_per_step"])
    except (KeyError, ValueError):
        return None


# ---------------------------------------------------------------------------
# multi-rank host logic (one process per GPU, weak scaling, no data-path
# collective): every rank steps its own full-size shard
# ---------------------------------------------------------------------------
def shard_seed(rank: int) -> int:
    """Seed of rank `rank`'s shard of the workload (shards differ)."""
    return 2 + rank


def max_over_ranks(x: float, dist, device) -> float:
    """The largest x over the ranks of the default process group."""
    import torch
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t)


def job_value(world: int, cells_per_rank: int, steps: int, total_ms: float) -> float:
    """Whole-job cell-updates/s: every rank's cells over the slowest rank's time."""
    return world * cells_per_rank * steps / (total_ms * 1e-3)


def bf16_peak() -> float:
    """Dense bf16 TFLOP/s: MEASURED_PEAKS.json (burst), else the fallback."""
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            d = json.load(f)
        if "bf16_tflops" in d:
            return float(d["bf16_tflops"])
    return 1900.0


def peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            d = json.load(f)
        for k in ("hbm_gbs", "hbm_GBs", "hbm"):
            if k in d:
                return float(d[k]), "measured"
    return FALLBACK_HBM_GBS, "fallback"


class ClockSampler:
    """nvidia-smi SM clocks and throttle reasons, sampled during a region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.p = None

    def __enter__(self):
        try:
            self.p = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.Q}", "--format=csv,noheader,nounits",
                 "-lms", "50", "-i", str(self.gpu)],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.p = None
        time.sleep(0.3)
        return self

    def __exit__(self, *exc):
        self.out = ""
        if self.p is not None:
            time.sleep(0.2)
            self.p.terminate()
            try:
                self.out, _ = self.p.communicate(timeout=5)
            except subprocess.TimeoutExpired:
                self.p.kill()
                self.out = ""

    def summary(self):
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in (self.out or "").splitlines():
            f = [x.strip() for x in line.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx.append(float(f[2]))
            except ValueError:
                continue
            for n, v in zip(names, f[5:9]):
                if v.lower() == "active":
                    reasons.add(n)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": [], "samples": 0}
        busy = sorted(sm)[len(sm) // 2:] or sm
        return {"sm_mhz": float(np.median(busy)), "sm_max_mhz": max(mx),
                "reasons": sorted(reasons), "samples": len(sm)}


def time_oracle_sample(idx_cpu, seed=2):
    """The FP64 oracle (as it stands) on a bounded sample of the workload's
    cells; returns (cell-updates/s, cells, seconds, threads, outputs)."""
    import torch

    import oracle
    from paper_2202_10647_gb300 import workloads as W

    sub = W.nitrogen_3d(*GRID, seed=seed, cells=torch.as_tensor(idx_cpu))
    n = sub.ncells
    osp = oracle.Species(sub.species.U, sub.species.l, sub.species.m)
    E = sub.E.double().numpy()
    N = sub.N[:, :n].double().numpy()
    lo, hi = sub.lo.numpy(), sub.hi.numpy()
    oracle.step(osp, E[:64], N[:, :64], 0.05, lo[:64], hi[:64])  # load + warm
    t0 = time.perf_counter()
    res = oracle.step(osp, E, N, 0.05, lo, hi)
    dt = time.perf_counter() - t0
    return n / dt, n, dt, oracle.num_threads(), res, sub


def sample_indices(total, n, seed=0):
    rng = np.random.default_rng(seed)
    return np.sort(rng.choice(total, size=min(n, total), replace=False))


def run_reference(args):
    """The oracle on this machine's host cores, on samples of the same workload."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    total = GRID[0] * GRID[1] * GRID[2]
    # size the per-step sample from a short probe so a step takes ~2-5 s
    rate, n, dt, threads, _, _ = time_oracle_sample(sample_indices(total, 20000, 99))
    per_step = int(min(total, max(20000, rate * 3.0)))
    times = []
    for s in range(args.warmup + args.steps):
        rate_s, n_s, dt_s, threads, _, _ = time_oracle_sample(sample_indices(total, per_step, s))
        if s >= args.warmup:
            times.append((n_s, dt_s))
    cells = sum(t[0] for t in times)
    secs = sum(t[1] for t in times)
    value = cells / secs
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": "cell-updates/s",
        "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": 1e3 * total / value, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": WORKLOAD, "cells": total, "dt_fs": 0.05,
                   "sample_cells_per_step": per_step},
        "cpu_baseline": {"value": value, "unit": "cell-updates/s", "cores": threads,
                         "kind": "oracle",
                         "sample": f"{per_step} random cells of the {total}-cell grid per step"},
        "e2e": {"value": value, "unit": "cell-updates/s", "h2d_bytes_per_step": 0,
                "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


def fp64_instructions(lmax, w):
    """FP64 instructions that the plain FP64 form cannot do without, per cell of largest
    W dt lmax and window width w (torch, any device): none below the first term of its series;
    else one for log2|E| and two for the exponent of each of the w-1 rates; and, up to
    W dt = 1/2, per term of the series (as many as keep the first one left out below 2e-17) a
    share of each state's sum, its outflow and its next term (the first and the last state one
    less), then the flows and what they add up to.  (The Bateman coefficients of the other
    cells are left out: a lower bound.)"""
    import math

    import torch
    lmax, w = lmax.double(), w.double()
    terms = torch.zeros_like(lmax)
    for k in range(1, 19):
        for width in range(2, 7):
            paths = sum(math.comb(k, j) for j in range(min(width - 1, k) + 1))
            thr = (2e-17 * math.factorial(k) / paths) ** (1.0 / k)
            terms += ((w == width) & (lmax > thr)).double()
    per_term = torch.clamp(3.0 * (w - 1.0) - 2.0, min=2.0)
    series = terms * per_term + 4.0 * (w - 1.0) - 1.0
    hot = 1.0 + 2.0 * (w - 1.0) + torch.where(lmax <= 0.5, series, torch.zeros_like(series))
    return torch.where((terms > 0) & (w >= 2), hot, torch.zeros_like(hot))


def _r(x, nd=4):
    return None if x is None else float(f"{x:.{nd}g}")


def summary_of(line):
    """ms per step, G cell-updates/s and roofline fraction of each form."""
    f = line["forms"]
    out = {"fp32_nitrogen": {"ms": _r(line["ms_per_step"]), "Gcells_s": _r(line["value"] / 1e9),
                             "frac_hbm": _r(line["roofline"]["frac"], 3)}}
    p = f.get("fp64_plain")
    if p:
        out["fp64_plain_nitrogen"] = {"ms": _r(p["ms_per_step"]), "Gcells_s": _r(p["value"] / 1e9),
                                      "frac_fp64_pipe": _r(p["roofline"]["frac"], 3)}
    b = f.get("batched_mixed_species")
    if b:
        out["batched_30M"] = {"ms": _r(b["ms_per_step"]), "Gcells_s": _r(b["value"] / 1e9),
                              "frac_hbm": _r(b["frac_of_hbm_peak"], 3),
                              "err": _r(b["max_abs_err_N_vs_oracle"], 2)}
        if b.get("roofline"):
            out["batched_30M"]["frac_issue"] = _r(b["roofline"]["frac"], 3)
    s = f.get("surrogate_argon")
    if s:
        out["surrogate_argon"] = {"ms": _r(s["ms_per_step"]),
                                  "plain_ms": _r(s["plain_fp32"]["ms_per_step"]),
                                  "plain_tuned_ms": _r((s.get("plain_fp32_autotuned") or {}).get(
                                      "ms_per_step")),
                                  "gain": _r(s["gain_vs_plain"], 3),
                                  "on_network": _r(s["cells_on_network_rates"], 3),
                                  "rate_err_median": _r((s.get("accuracy") or {}).get(
                                      "median_rel_rate_error"), 3)}
    k = f.get("krypton_beams_50_steps_graph")
    if k:
        out["krypton_50_steps"] = {"ms_with_check": _r(k["ms_per_50_steps"]),
                                   "ms_steps_only": _r(k["ms_per_50_steps_steps_only"]),
                                   "ms_adaptive": _r(k["adaptive_window_steps_only"]["ms_per_50_steps"]),
                                   "ms_surrogate": _r((k.get("surrogate_form") or {}).get(
                                       "ms_per_50_steps")),
                                   "ms_full_check": _r(k["ms_per_50_steps_full_check_each_step"]),
                                   "max_sum_err": _r(k["max_abs_sum_N_minus_1"]["after_step_50"], 2)}
    if line.get("e2e"):
        out["e2e_ms"] = _r(line["e2e"]["ms_per_step"])
    return out


def main():
    args = parse()
    if args.impl == "reference":
        run_reference(args)
        return

    import torch
    import torch.distributed as dist

    from paper_2202_10647_gb300 import ionize
    from paper_2202_10647_gb300 import workloads as W

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if world > 1:
        dist.init_process_group("nccl", device_id=dev)

    # -- inputs (resident in HBM before timing starts) ----------------------
    wl = W.nitrogen_3d(*GRID, seed=shard_seed(rank), device=dev)
    n = wl.ncells
    sp = ionize.Species(wl.species.U, wl.species.l, wl.species.m)
    N0, lo0, hi0 = wl.N.clone(), wl.lo.clone(), wl.hi.clone()
    N, lo, hi, E = wl.N, wl.lo, wl.hi, wl.E
    dne = torch.empty(n, dtype=torch.float32, device=dev)
    ws = ionize.workspace(n, ionize.ION_F32, dev)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)  # > L2 (129 MB)
    w = (hi0.long() - lo0.long() + 1)
    alg_bytes = int(W.window_bytes_per_cell(lo0, hi0).sum())
    mean_w = float(w.double().mean())
    stream = torch.cuda.current_stream(dev)

    def restore():
        N.copy_(N0)
        lo.copy_(lo0)
        hi.copy_(hi0)
        flush.zero_()

    def timed_loop(K, Wm, fn):
        evs = []
        for s in range(Wm + K):
            restore()
            a = torch.cuda.Event(enable_timing=True)
            b = torch.cuda.Event(enable_timing=True)
            a.record(stream)
            fn()
            b.record(stream)
            if s >= Wm:
                evs.append((a, b))
        torch.cuda.synchronize()
        return [a.elapsed_time(b) for a, b in evs]

    def step_f32():
        ionize.step(sp, E, N, lo, hi, 0.05, dne, ws=ws)

    # sampled cells for the accuracy report (inputs copied before the step)
    idx = torch.tensor(sample_indices(n, 4000, 1), device=dev)

    # -- timed region: the metric -------------------------------------------
    timed_loop(0, args.warmup, step_f32)
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    with ClockSampler(local) as clk:
        t_step = timed_loop(args.steps, 0, step_f32)
    torch.cuda.synchronize()
    fb_cells, bad = 0, 0
    restore()
    step_f32()
    torch.cuda.synchronize()
    fb_cells, bad = ionize.counters(ws)
    stiff = ionize.stiff_cells(ws)
    total_ms = float(sum(t_step))
    if world > 1:
        total_ms = max_over_ranks(total_ms, dist, dev)
        dist.barrier()
    ms_per_step = total_ms / args.steps
    value = job_value(world, n, args.steps, total_ms)
    # the roofline is taken over the whole step (its three kernels and the
    # counter reset): algorithmic bytes of one step / measured step time
    main_ms = float(np.mean(t_step))
    peak, peak_kind = peaks()
    achieved = alg_bytes / (main_ms * 1e-3) / 1e9

    # -- the plain FP64 form on the same inputs ------------------------------
    E64 = E.double()
    N64_0 = N0.double()
    N64 = N64_0.clone()
    dne64 = torch.empty(n, dtype=torch.float64, device=dev)
    ws64 = ionize.workspace(n, ionize.ION_F64_PLAIN, dev)

    def step_f64():
        ionize.step(sp, E64, N64, lo, hi, 0.05, dne64, ws=ws64, flags=ionize.ION_F64_PLAIN)

    def restore64():
        N64.copy_(N64_0)
        lo.copy_(lo0)
        hi.copy_(hi0)
        flush.zero_()

    k64 = max(3, min(20, args.steps // 10))
    ev64 = []
    for s in range(2 + k64):
        restore64()
        a = torch.cuda.Event(enable_timing=True)
        b = torch.cuda.Event(enable_timing=True)
        a.record(stream)
        step_f64()
        b.record(stream)
        if s >= 2:
            ev64.append((a, b))
    torch.cuda.synchronize()
    ms64 = float(np.mean([a.elapsed_time(b) for a, b in ev64]))
    bytes64 = int(W.window_bytes_per_cell(lo0, hi0, elem=8).sum())
    # the FP64 form is bound by the FP64 pipe: the instructions that its cells
    # need, counted on a sample, against the measured FP64 multiply-add rate
    pk = ionize.measure_peaks()
    pick = torch.randint(0, n, (1 << 20,), generator=torch.Generator(device=dev).manual_seed(5),
                         device=dev)
    W64 = ionize.rates(sp, E64[pick].contiguous(), 0, sp.Z) * 0.05
    k_ = torch.arange(sp.Z, device=dev)[:, None]
    W64 *= (k_ >= lo0[pick].long()) & (k_ < hi0[pick].long())
    inst64 = float(fp64_instructions(W64.max(0).values, w[pick]).mean()) * n
    del W64
    # FP64 vs FP32 outputs on the same inputs (one step each)
    restore64()
    step_f64()
    restore()
    step_f32()
    torch.cuda.synchronize()
    diff_32_64 = float((N[:, :n].double() - N64[:, :n]).abs().max())
    del E64, N64_0, N64, dne64

    # -- batched form: N (20M), Ar-like (8M), Kr-like (2M) cells in one launch -
    batched = None
    if not args.no_batched:
        bjobs_wl = W.mixed_batch(scale=1.0, seed=3, device=dev)
        bsp = [ionize.Species(w_.species.U, w_.species.l, w_.species.m) for w_ in bjobs_wl]
        pristine = [(w_.N.clone(), w_.lo.clone(), w_.hi.clone()) for w_ in bjobs_wl]
        bdne = [torch.empty(w_.ncells, device=dev) for w_ in bjobs_wl]
        bjobs = [(sp_, w_.E, w_.N, w_.lo, w_.hi, d_) for sp_, w_, d_ in zip(bsp, bjobs_wl, bdne)]
        bws = ionize.batched_workspace(bjobs)

        def brestore():
            for w_, (n0, l0, h0) in zip(bjobs_wl, pristine):
                w_.N.copy_(n0)
                w_.lo.copy_(l0)
                w_.hi.copy_(h0)
            flush.zero_()

        # the autotuner steps the arrays (each of its launches starts from the
        # state the previous one left): its pick and the two default shapes
        # are then timed again from the restored state, and the fastest kept
        tuned, tune_ms = ionize.autotune(bjobs, 0.05, ws=bws, reps=3)
        cands = [tuned] + [ionize.LaunchShape(*c) for c in ((2, 8, 0), (1, 8, 0))
                           if c != (tuned.cells_per_lane, tuned.warps_per_block,
                                    tuned.blocks_per_sm)]
        cand_ms = []
        for c_ in cands:
            ts_ = []
            for s_ in range(4):
                brestore()
                a_ = torch.cuda.Event(enable_timing=True)
                b_ = torch.cuda.Event(enable_timing=True)
                a_.record(stream)
                ionize.step_batched(bjobs, 0.05, ws=bws, shape=c_)
                b_.record(stream)
                if s_ >= 1:
                    ts_.append((a_, b_))
            torch.cuda.synchronize()
            cand_ms.append(float(np.mean([a_.elapsed_time(b_) for a_, b_ in ts_])))
        shape = cands[int(np.argmin(cand_ms))]
        bt = []
        for s_ in range(3 + max(5, args.steps // 5)):
            brestore()
            a_ = torch.cuda.Event(enable_timing=True)
            b_ = torch.cuda.Event(enable_timing=True)
            a_.record(stream)
            ionize.step_batched(bjobs, 0.05, ws=bws, shape=shape)
            b_.record(stream)
            if s_ >= 3:
                bt.append((a_, b_))
        torch.cuda.synchronize()
        bms = float(np.mean([a_.elapsed_time(b_) for a_, b_ in bt]))
        # the step again in the shape of the committed instruction counts
        # (the issue roofline's), when the autotuner picked another
        rshape = recorded_issue_shape()
        bms_rec = bms
        if rshape and rshape != (shape.cells_per_lane, shape.warps_per_block,
                                 shape.blocks_per_sm):
            bt = []
            for s_ in range(3 + max(5, args.steps // 5)):
                brestore()
                a_ = torch.cuda.Event(enable_timing=True)
                b_ = torch.cuda.Event(enable_timing=True)
                a_.record(stream)
                ionize.step_batched(bjobs, 0.05, ws=bws, shape=rshape)
                b_.record(stream)
                if s_ >= 3:
                    bt.append((a_, b_))
            torch.cuda.synchronize()
            bms_rec = float(np.mean([a_.elapsed_time(b_) for a_, b_ in bt]))
        bcells = sum(w_.ncells for w_ in bjobs_wl)
        bbytes = sum(int(W.window_bytes_per_cell(l0, h0).sum()) for (_, l0, h0) in pristine)
        # accuracy on sampled cells of each species
        bacc = 0.0
        if rank == 0:
            import oracle
            brestore()
            samples = []
            for w_ in bjobs_wl:
                ix = torch.tensor(sample_indices(w_.ncells, 2000, 5), device=dev)
                samples.append((ix, w_.E[ix].double().cpu().numpy(),
                                w_.N[:, ix].double().cpu().numpy(), w_.lo[ix].cpu().numpy(),
                                w_.hi[ix].cpu().numpy()))
            ionize.step_batched(bjobs, 0.05, ws=bws, shape=shape)
            torch.cuda.synchronize()
            for w_, (ix, Es_, Ns_, ls_, hs_) in zip(bjobs_wl, samples):
                osp_ = oracle.Species(w_.species.U, w_.species.l, w_.species.m)
                No_, _, _, _ = oracle.step(osp_, Es_, Ns_, 0.05, ls_, hs_)
                bacc = max(bacc, float(np.abs(w_.N[:, ix].double().cpu().numpy() - No_).max()))
        batched = {"value": bcells / (bms * 1e-3), "ms_per_step": bms, "cells": bcells,
                   "species": "N 20M + Ar-like 8M + Kr-like 2M",
                   "achieved_GBs": bbytes / (bms * 1e-3) / 1e9,
                   "frac_of_hbm_peak": bbytes / (bms * 1e-3) / 1e9 / peaks()[0],
                   "launch_shape": {"cells_per_lane": shape.cells_per_lane,
                                    "warps_per_block": shape.warps_per_block,
                                    "blocks_per_sm": shape.blocks_per_sm},
                   "shape_choice": {"autotuned": [tuned.cells_per_lane, tuned.warps_per_block,
                                                  tuned.blocks_per_sm],
                                    "candidates_ms": {f"{c_.cells_per_lane},{c_.warps_per_block},"
                                                      f"{c_.blocks_per_sm}": round(m_, 4)
                                                      for c_, m_ in zip(cands, cand_ms)}},
                   "max_abs_err_N_vs_oracle": bacc,
                   "ms_per_step_at_recorded_shape": bms_rec}
        del bjobs, bjobs_wl, pristine, bws

    # -- surrogate form: Ar-like cells, rates from the tensor-core network ----
    surrogate = None
    if not args.no_surrogate:
        from paper_2202_10647_gb300 import surrogate as S
        sd4 = W.argon_like()
        sp4 = ionize.Species(sd4.U, sd4.l, sd4.m)
        t0 = time.time()
        net4, tr4, bound4 = S.build(sp4)
        torch.cuda.synchronize()
        train_s = time.time() - t0
        n4 = 33_554_432
        wl4 = W.ladder_cells(sd4, n4, 4, device=dev)
        N40, lo40, hi40 = wl4.N.clone(), wl4.lo.clone(), wl4.hi.clone()
        dne4 = torch.empty(n4, device=dev)
        ws4 = ionize.workspace(n4)

        def r4():
            wl4.N.copy_(N40)
            wl4.lo.copy_(lo40)
            wl4.hi.copy_(hi40)
            flush.zero_()

        def t4(fn, reps):
            ts_ = []
            for r_ in range(reps + 3):
                r4()
                a_ = torch.cuda.Event(enable_timing=True)
                b_ = torch.cuda.Event(enable_timing=True)
                a_.record(stream)
                fn()
                b_.record(stream)
                if r_ >= 3:
                    ts_.append((a_, b_))
            torch.cuda.synchronize()
            return float(np.mean([a_.elapsed_time(b_) for a_, b_ in ts_]))

        reps4 = max(5, min(30, args.steps // 10))
        t_plain4 = t4(lambda: ionize.step(sp4, wl4.E, wl4.N, wl4.lo, wl4.hi, 0.05, dne4, ws=ws4),
                      reps4)
        t_net4 = t4(lambda: net4.step(wl4.E, wl4.N, wl4.lo, wl4.hi, 0.05, dne4, ws=ws4), reps4)
        n_net4, n_plain4, tmo4 = ionize.surrogate_counters(ws4)
        # the same plain step with the launch shape the library's autotuner
        # picks for these cells (the autotuner steps the arrays: restored by t4;
        # after the surrogate counters are read: it reuses their workspace)
        # (its pick and the two default shapes timed again from the restored
        # state, the fastest kept: the autotuner's launches step the arrays in
        # turn)
        job4 = [(sp4, wl4.E, wl4.N, wl4.lo, wl4.hi, dne4)]
        shape4, _ = ionize.autotune(job4, 0.05, ws=ws4, reps=3)
        t_tuned4 = t4(lambda: ionize.step_batched(job4, 0.05, ws=ws4, shape=shape4), reps4)
        for c4 in ((1, 8, 0), (2, 8, 0)):
            if (shape4.cells_per_lane, shape4.warps_per_block, shape4.blocks_per_sm) == c4:
                continue
            alt4 = ionize.LaunchShape(*c4)
            t_alt4 = t4(lambda: ionize.step_batched(job4, 0.05, ws=ws4, shape=alt4), reps4)
            if t_alt4 < t_tuned4:
                shape4, t_tuned4 = alt4, t_alt4
        acc4 = None
        if rank == 0:
            import oracle
            ix4 = torch.tensor(sample_indices(n4, 4000, 6), device=dev)
            r4()
            Es4 = wl4.E[ix4].double().cpu().numpy()
            Ns4 = wl4.N[:, ix4].double().cpu().numpy()
            ls4, hs4 = wl4.lo[ix4].cpu().numpy(), wl4.hi[ix4].cpu().numpy()
            net4.step(wl4.E, wl4.N, wl4.lo, wl4.hi, 0.05, dne4, ws=ws4)
            Nnet = wl4.N[:, ix4].double().cpu().numpy()
            r4()
            ionize.step(sp4, wl4.E, wl4.N, wl4.lo, wl4.hi, 0.05, dne4, ws=ws4)
            Npl = wl4.N[:, ix4].double().cpu().numpy()
            osp4 = oracle.Species(sd4.U, sd4.l, sd4.m)
            No4, _, _, _ = oracle.step(osp4, Es4, Ns4, 0.05, ls4, hs4)
            Wn4 = net4.rates(wl4.E[ix4].contiguous()).double().cpu().numpy()
            Wo4 = oracle.rates(osp4, Es4, 0, sd4.Z)
            big4 = Wo4 * 0.05 > 1e-12
            rel4 = np.abs(Wn4[big4] / Wo4[big4] - 1.0)
            acc4 = {"max_rel_rate_error": float(rel4.max()),
                    "median_rel_rate_error": float(np.median(rel4)),
                    "rate_error_over": "states with W dt > 1e-12 of 4000 sampled cells",
                    "max_abs_err_N_vs_oracle_surrogate_form": float(np.abs(Nnet - No4).max()),
                    "max_abs_err_N_vs_oracle_plain_fp32": float(np.abs(Npl - No4).max())}
        surrogate = {"value": n4 / (t_net4 * 1e-3), "ms_per_step": t_net4,
                     "plain_fp32": {"value": n4 / (t_plain4 * 1e-3), "ms_per_step": t_plain4},
                     "plain_fp32_autotuned": {
                         "value": n4 / (t_tuned4 * 1e-3), "ms_per_step": t_tuned4,
                         "shape": [shape4.cells_per_lane, shape4.warps_per_block,
                                   shape4.blocks_per_sm]},
                     "gain_vs_plain": t_plain4 / t_net4,
                     "cells": n4, "species": "Ar-like (Z=18)",
                     "network": "1-64-64-18 GELU, weights and activations as bf16 pairs, FP32 accumulation (tcgen05)",
                     "train": {"seconds": train_s, "steps": tr4.steps, "pairs": 1 << 20,
                               "final_loss": tr4.losses[-1][1]},
                     "pop_tol": 1e-6,
                     # the network's work per cell: 128 GELUs (one SFU tanh
                     # each) and 2 (64*64 + 64*Z) tensor flops of the method
                     # (its Z outputs; the tensor cores run three bf16
                     # products per pair and pad the outputs to 32 columns)
                     "roofline": {
                         "bound": "alu",
                         "achieved": 128 * n4 / (t_net4 * 1e-3),
                         "peak": pk["sfu_tanh_per_s"],
                         "unit": "SFU tanh/s",
                         "frac": 128 * n4 / (t_net4 * 1e-3) / pk["sfu_tanh_per_s"],
                         "peak_source": "measured (ion_measure_peaks)",
                         "tensor_TFLOPs": 2 * (64 * 64 + 64 * sd4.Z) * n4 / (t_net4 * 1e-3) / 1e12,
                         "tensor_frac_of_bf16_peak": 2 * (64 * 64 + 64 * sd4.Z) * n4
                         / (t_net4 * 1e-3) / 1e12 / bf16_peak(),
                         "note": "whole surrogate step (network kernel + record kernel)"},
                     "cells_on_network_rates": n_net4 / n4,
                     "cells_on_eq1_rates": n_plain4 / n4, "timeouts": tmo4,
                     "accuracy": acc4}
        del wl4, N40, lo40, hi40, dne4, ws4

    # -- Kr-like 512x512x256 cells, 50 steps captured in one CUDA graph -------
    krypton = None
    if not args.no_krypton:
        from paper_2202_10647_gb300 import multistep
        kgrid = (256, 512, 512)
        kn = kgrid[0] * kgrid[1] * kgrid[2]
        A_, B_ = W.krypton_beam_terms(*kgrid, device=dev)
        S_ = W.krypton_scale(A_)
        kfields = [W.krypton_field(A_, B_, s_ * 0.05, S_) for s_ in range(50)]
        del A_, B_
        kwl = W.krypton_initial(kn, device=dev)
        ksp = ionize.Species(kwl.species.U, kwl.species.l, kwl.species.m)
        kdne = torch.empty(kn, device=dev)
        kws = ionize.workspace(kn)
        graphs = {name: multistep.StepGraph(ksp, kfields, kwl.N, kwl.lo, kwl.hi, kdne, 0.05,
                                            ws=kws, conservation=chk)
                  for name, chk in (("with_check", "fused"), ("with_full_check", "full"),
                                    ("steps_only", False))}
        graphs["adaptive_window"] = multistep.StepGraph(
            ksp, kfields, kwl.N, kwl.lo, kwl.hi, kdne, 0.05, ws=kws, conservation=False,
            window=dict(w_min=2, w_max=6, eps_grow=1e-6))
        knet = None
        if not args.no_surrogate:
            from paper_2202_10647_gb300 import surrogate as S
            knet, _, _ = S.build(ksp)
            graphs["surrogate_with_check"] = multistep.StepGraph(
                ksp, kfields, kwl.N, kwl.lo, kwl.hi, kdne, 0.05, ws=kws, conservation=True,
                surrogate=knet)

        def kreset():
            kwl.N.zero_()
            kwl.N[0, :kn] = 1.0
            kwl.lo.zero_()
            kwl.hi.fill_(3)

        kres, kwidth = {}, {}
        for name, g_ in graphs.items():
            ts_ = []
            for r_ in range(4):
                kreset()
                a_ = torch.cuda.Event(enable_timing=True)
                b_ = torch.cuda.Event(enable_timing=True)
                a_.record(stream)
                g_.replay()
                b_.record(stream)
                torch.cuda.synchronize()
                if r_ >= 1:
                    ts_.append(a_.elapsed_time(b_))
            kres[name] = float(np.median(ts_))
            kwidth[name] = float((kwl.hi.double() - kwl.lo.double() + 1).mean())
        cons = graphs["with_check"].cons.cpu().numpy()
        cons_full = graphs["with_check"].cons_full.cpu().numpy()
        cons_each = graphs["with_full_check"].cons.cpu().numpy()
        ksur = None
        if "surrogate_with_check" in graphs:
            kc = graphs["surrogate_with_check"].cons.cpu().numpy()
            ksur = {"value": 50 * kn / (kres["surrogate_with_check"] * 1e-3),
                    "ms_per_50_steps": kres["surrogate_with_check"],
                    "max_abs_sum_N_minus_1": float(kc.max()),
                    "network": "1-64-64-36 GELU, weights and activations as bf16 pairs, FP32 accumulation (tcgen05)"}
        krypton = {"value": 50 * kn / (kres["with_check"] * 1e-3),
                   "ms_per_50_steps": kres["with_check"],
                   "value_steps_only": 50 * kn / (kres["steps_only"] * 1e-3),
                   "ms_per_50_steps_steps_only": kres["steps_only"],
                   "cells": kn, "grid": list(kgrid), "species": "Kr-like (Z=36), 37 planes",
                   "field": "16 seeded Gaussian beams, lambda 0.8 um, 6000 GV/m peak at t=0",
                   "graph": "50 x ion_step with its own conservation measure "
                            "(ION_CONSERVATION_CHECK), ion_conservation over all 37 "
                            "planes after steps 1 and 50, in one CUDA graph",
                   "max_abs_sum_N_minus_1": {"after_step_1": float(cons_full[0]),
                                             "after_step_50": float(cons_full[1]),
                                             "max_step_change": float(cons.max()),
                                             "sum_of_step_changes": float(cons.sum())},
                   "ms_per_50_steps_full_check_each_step": kres["with_full_check"],
                   "full_check_each_step_max_abs_sum_N_minus_1": float(cons_each.max()),
                   "windows_slid_fraction": float((kwl.lo > 0).double().mean()),
                   "surrogate_form": ksur,
                   "adaptive_window_steps_only": {
                       "policy": "w_min 2, w_max 6, eps_grow 1e-6",
                       "ms_per_50_steps": kres["adaptive_window"],
                       "value": 50 * kn / (kres["adaptive_window"] * 1e-3),
                       "mean_width_after_50_steps": kwidth["adaptive_window"],
                       "fixed_mean_width_after_50_steps": kwidth["steps_only"]}}
        del graphs, kfields, kwl, kws, kdne, knet

    # -- end to end through host buffers -------------------------------------
    e2e = None
    if not args.no_e2e:
        hE = E.cpu().pin_memory()
        hN = N0.cpu().pin_memory()
        hlo = lo0.cpu().pin_memory()
        hhi = hi0.cpu().pin_memory()
        oN = torch.empty_like(hN).pin_memory()
        olo = torch.empty_like(hlo).pin_memory()
        ohi = torch.empty_like(hhi).pin_memory()
        odne = torch.empty(n, dtype=torch.float32).pin_memory()

        def e2e_sequential():
            E.copy_(hE, non_blocking=True)
            N.copy_(hN, non_blocking=True)
            lo.copy_(hlo, non_blocking=True)
            hi.copy_(hhi, non_blocking=True)
            ionize.step(sp, E, N, lo, hi, 0.05, dne, ws=ws)
            oN.copy_(N, non_blocking=True)
            olo.copy_(lo, non_blocking=True)
            ohi.copy_(hi, non_blocking=True)
            odne.copy_(dne, non_blocking=True)

        # the same step over 16 chunks of cells on three streams: inputs of
        # chunk i+1 go up while chunk i is stepped and chunk i-1 comes down
        sH, sC, sD = (torch.cuda.Stream(dev) for _ in range(3))
        nch = max(1, args.e2e_chunks)
        bounds = [(n * i // nch) // 256 * 256 for i in range(nch)] + [n]
        evs = [(torch.cuda.Event(), torch.cuda.Event()) for _ in range(nch)]
        start_ev = torch.cuda.Event()

        def e2e_pipelined():
            start_ev.record(stream)
            for s_ in (sH, sC, sD):
                s_.wait_event(start_ev)
            for i in range(nch):
                c0, c1 = bounds[i], bounds[i + 1]
                with torch.cuda.stream(sH):
                    ionize.copy_cells(E, hE, c0, c1 - c0)
                    ionize.copy_cells(N, hN, c0, c1 - c0)  # every plane, one strided copy
                    ionize.copy_cells(lo, hlo, c0, c1 - c0)
                    ionize.copy_cells(hi, hhi, c0, c1 - c0)
                    evs[i][0].record(sH)
                sC.wait_event(evs[i][0])
                with torch.cuda.stream(sC):
                    ionize.step(sp, E, N, lo, hi, 0.05, dne, ws=ws, offset=c0, ncells=c1 - c0)
                    evs[i][1].record(sC)
                sD.wait_event(evs[i][1])
                with torch.cuda.stream(sD):
                    ionize.copy_cells(oN, N, c0, c1 - c0)
                    ionize.copy_cells(olo, lo, c0, c1 - c0)
                    ionize.copy_cells(ohi, hi, c0, c1 - c0)
                    ionize.copy_cells(odne, dne, c0, c1 - c0)
            stream.wait_stream(sD)

        ke = max(5, min(20, args.steps // 15))

        # each step timed on its own; the median, since the host link is
        # shared with the machine's other GPUs and their jobs' copies
        def e2e_time(fn):
            for _ in range(2):
                fn()
            torch.cuda.synchronize()
            ev_ = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
                   for _ in range(ke)]
            for a, b in ev_:
                a.record(stream)
                fn()
                b.record(stream)
            torch.cuda.synchronize()
            t_ = [a.elapsed_time(b) for a, b in ev_]
            return float(np.median(t_)), float(np.min(t_)), float(np.max(t_))

        e_seq_ms, e_seq_min, e_seq_max = e2e_time(e2e_sequential)
        e_ms, e_min, e_max = e2e_time(e2e_pipelined)
        # the pipelined run's outputs are those of one whole-grid step
        e2e_sequential()
        torch.cuda.synchronize()
        ref_out = oN.clone()
        e2e_pipelined()
        torch.cuda.synchronize()
        e2e_same = bool(torch.equal(ref_out, oN))
        h2d = hE.numel() * 4 + hN.numel() * 4 + 2 * n
        d2h = oN.numel() * 4 + 2 * n + 4 * n
        e2e = {"value": n / (e_ms * 1e-3), "unit": "cell-updates/s",
               "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h,
               "ms_per_step": e_ms,
               "how": f"{nch} cell chunks, host-to-device, step and device-to-host on three "
                      "streams (pinned host buffers; ion_copy_cells moves all planes of a "
                      "chunk in one strided copy)",
               "steps_timed": ke, "ms_min_max": [e_min, e_max],
               "sequential_ms_per_step": e_seq_ms, "sequential_ms_min_max": [e_seq_min, e_seq_max],
               "pipelined_output_equals_sequential": e2e_same}
        del hE, hN, oN

    # -- accuracy on sampled cells and the CPU oracle baseline ---------------
    cpu = None
    acc = None
    if rank == 0:
        import oracle
        restore()
        Es, Ns = E[idx].double().cpu().numpy(), N[:, idx].double().cpu().numpy()
        los, his = lo[idx].cpu().numpy(), hi[idx].cpu().numpy()
        step_f32()
        torch.cuda.synchronize()
        osp = oracle.Species(wl.species.U, wl.species.l, wl.species.m)
        No, _, _, dneo = oracle.step(osp, Es, Ns, 0.05, los, his)
        acc = {"max_abs_err_N_vs_oracle": float(np.abs(N[:, idx].double().cpu().numpy() - No).max()),
               "max_abs_err_dne_vs_oracle": float(np.abs(dne[idx].double().cpu().numpy() - dneo).max()),
               "sample_cells": int(idx.numel()),
               "max_conservation_err": float((N[:, :n].double().sum(0) - N0[:, :n].double().sum(0)).abs().max()),
               "fp32_vs_fp64_form_max_abs": diff_32_64}
        if not args.no_cpu_baseline:
            total = n
            rate, _, dtp, threads, _, _ = time_oracle_sample(sample_indices(total, 20000, 99))
            ns = int(min(total, max(20000, rate * 12.0)))
            rate, ns, dts, threads, _, _ = time_oracle_sample(sample_indices(total, ns, 98))
            cpu = {"value": rate, "unit": "cell-updates/s", "cores": threads, "kind": "oracle",
                   "sample": f"{ns} random cells of the {total}-cell grid, one step ({dts:.1f} s)"}

    if rank != 0:
        return
    clocks = clk.summary()
    if batched is not None:
        batched["roofline"] = batched_issue_roofline(
            batched["ms_per_step_at_recorded_shape"], clocks.get("sm_mhz") or clocks.get("sm_max_mhz"),
            torch.cuda.get_device_properties(dev).multi_processor_count)
    line = {
        "metric": METRIC, "value": value, "unit": "cell-updates/s", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_per_step,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
        "data": "synthetic",
        "config": {"workload": WORKLOAD, "grid": list(GRID), "cells_per_gpu": n,
                   "species": "N (Z=7)", "dt_fs": 0.05, "mean_window_width": mean_w,
                   "l2": "flushed between timed steps (256 MB write) and inputs > L2",
                   "form": "FP32 + FP64 coefficients for |W_i-W_j| < 1e-3 max(W_i,W_j)"},
        "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                     "frac": achieved / peak, "traffic": recorded_traffic(),
                     "kernel": "ion_step (ion_lean_kernel + ion_stiff_kernel + ion_fb_kernel)",
                     "peak_source": peak_kind,
                     "algorithmic_bytes_per_launch": alg_bytes, "kernel_ms": main_ms},
        "forms": {
            "fp32_fp64fallback": {"value": value, "ms_per_step": ms_per_step,
                                  "fp64_coefficient_cells": fb_cells,
                                  "second_kernel_cells": stiff},
            "fp64_plain": {"value": n / (ms64 * 1e-3), "ms_per_step": ms64,
                           "achieved_GBs": bytes64 / (ms64 * 1e-3) / 1e9,
                           "roofline": {"bound": "alu",
                                        "achieved": inst64 / (ms64 * 1e-3),
                                        "peak": pk["fp64_flops"] / 2,
                                        "unit": "FP64 instructions/s",
                                        "frac": inst64 / (ms64 * 1e-3) / (pk["fp64_flops"] / 2),
                                        "fp64_instructions_per_cell": inst64 / n,
                                        "peak_source": "measured FP64 multiply-add rate "
                                                       "(ion_measure_peaks)"}},
            "batched_mixed_species": batched,
            "krypton_beams_50_steps_graph": krypton,
            "surrogate_argon": surrogate,
        },
        "accuracy": acc,
        "peaks_measured": pk,
        # the header's clearing, the streaming, record and queue kernels
        "gpu_launches": 4 * args.steps,
        "clocks": clocks,
        "cpu_baseline": cpu,
        "e2e": e2e,
    }
    # the headline numbers of every form again, compact and last on the line
    # (a reader of the line's tail sees them all)
    line["summary"] = summary_of(line)
    print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
