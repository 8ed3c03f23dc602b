"""Throughput benchmark of the MBBP-LD hot path on GB300.

Workload (one "step"): the [[144,12,12]] bivariate bicycle code under
code-capacity depolarizing noise at p in {0.02, 0.04, 0.06, 0.08}; for every p,
SHOTS fresh shots are sampled on the GPU, the X part is decoded with the R=16
representations of H_Z and the Z part with those of H_X (100 iterations,
normalized min-sum, alpha = 0.625, FP32), FWS selects, and the logical judge
counts failures.  Every stage runs in the library's kernels through the C ABI;
each decode call (persistent BP kernel + FWS) is captured once into a CUDA
graph and replayed every step.

Output: one JSON line (rank 0).  ``value`` = depolarizing shots per second
(both error types decoded) with everything resident in HBM; ``e2e`` = the same
metric through mbbp_decode with pinned host syndromes copied in and estimates
copied out inside the timed region.  ``--impl reference`` times the CPU
oracle instead (the slow plain restatement of the method), on a bounded
sample of the same workload.

Multi-GPU (torchrun): rank r decodes its own shot range each step; the only
exchange is the failure / work counters, summed once after timing.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

CODE = "bb144"
P_LIST = (0.02, 0.04, 0.06, 0.08)
R = 16
ITERS = 100
ALPHA = 0.625
SEED = 20260515
OPS_PER_EDGE_UPDATE = 10  # algorithmic ALU operations per edge-update (min-sum flooding)
# Of those, 7 (|q|, three min1/min2 updates, sign parity, output select, sign
# apply) are min/max and logic operations, which a GB300 SM executes on its
# alu pipe at 64 lanes per clock, and 3 (alpha product, posterior and
# extrinsic adds) FP32 multiplies and adds on its fma pipe at 128 lanes per
# clock; the SM issues 128 lanes per clock (pipe widths confirmed by the
# library's throughput probes, mbbp_probe).
ALU_OPS, FMA_OPS = 7, 3
ALU_LANES, FMA_LANES, ISSUE_LANES = 64, 128, 128
EDGE_UPDATES_PER_CLK_SM = min(ALU_LANES / ALU_OPS, FMA_LANES / FMA_OPS, ISSUE_LANES / OPS_PER_EDGE_UPDATE)
# DRAM bytes per shot of the BP kernel: one ncu capture of a 100k-shot launch
# of the current kernel and layout (profiles/kernels_current.md: 7.315 MB read
# + 45 KB written); set to None whenever the kernel changes until it is
# captured again
DRAM_BYTES_PER_SHOT = (7.314944e6 + 4.5312e4) / 100000
WORKLOAD = "[[144,12,12]] BB, depolarizing p in {0.02,0.04,0.06,0.08}, X and Z decoded, R=16, 100 iters"


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="bb144", choices=["bb144", "mixed", "learned", "paper", "wms", "gb882"],
                    help="bb144: the headline configuration; mixed: [[72]]/[[144]]/[[288]] in one "
                         "persistent graph-captured launch vs plain per-code launches")
    ap.add_argument("--shots", type=int, default=None,
                    help="bb144: shots per p per step per GPU (default 1e6); mixed: shots per step (default 3e5)")
    ap.add_argument("--cpu-seconds", type=float, default=15.0, help="CPU baseline budget")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-extra", action="store_true",
                    help="bb144: skip the mixed-batch and length-882 legs reported beside the headline")
    ap.add_argument("--train-steps", type=int, default=300, help="learned: training steps")
    ap.add_argument("--p", type=float, default=None, help="gb882: a single error rate")
    ap.add_argument("--wms", action="store_true", help="gb882: also the weighted decoder at its initial weights")
    ap.add_argument("--train-batch", type=int, default=1024, help="learned: shots per training step")
    return ap.parse_args()


def read_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            return json.load(f), "measured"
    return {"hbm_gbs": 6800.0, "sm_max_mhz": 2070.0}, "fallback"


class ClockSampler:
    """nvidia-smi clock / throttle samples during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
        return self

    def __exit__(self, *exc):
        self.out = ""
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.out, _ = self.proc.communicate(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
                self.out, _ = self.proc.communicate()

    def summary(self):
        rows = []
        for line in (self.out or "").strip().splitlines():
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                rows.append((float(parts[1]), float(parts[2]), parts[5:9]))
            except ValueError:
                continue
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unavailable"], "samples": 0}
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        seen = sorted({names[i] for _, _, r in rows for i, v in enumerate(r) if v.lower() == "active"})
        loaded = [c for c, _, _ in rows]
        return {"sm_mhz": statistics.median(loaded), "sm_max_mhz": max(m for _, m, _ in rows),
                "reasons": seen, "samples": len(rows)}


def _oracle_rate(seconds: float, threads: int, precision: str):
    """Shots/s of the oracle (as it stands) on `threads` host threads over a
    bounded sample of the workload (shots taken round-robin over p)."""
    import concurrent.futures as cf

    import oracle
    from paper_2605_14170_gb300.inputs import named_code

    code = named_code(CODE)
    n = code.n
    sets = {"HZ": oracle.collect_subtrees(code.HZ, R, SEED), "HX": oracle.collect_subtrees(code.HX, R, SEED + 1)}
    chunk = 4

    def work(k):
        p = P_LIST[k % len(P_LIST)]
        first = 10_000_000 + chunk * k
        ex, ez = oracle.sample(SEED, first, chunk, n, p, "depolarizing")
        pm = 2 * p / 3
        llr = np.full(n, np.log((1 - pm) / pm))
        for H, e, key in ((code.HZ, ex, "HZ"), (code.HX, ez, "HX")):
            s = oracle.syndrome(H, e)
            oracle.mbbp_decode(H, sets[key], s, llr, ITERS, ALPHA, precision=precision)
        return chunk

    done = 0
    t0 = time.perf_counter()
    k = 0
    with cf.ThreadPoolExecutor(max_workers=threads) as ex:
        futs = set()
        while time.perf_counter() - t0 < seconds or futs:
            while len(futs) < threads and time.perf_counter() - t0 < seconds:
                futs.add(ex.submit(work, k))
                k += 1
            finished, futs = cf.wait(futs, return_when=cf.FIRST_COMPLETED)
            done += sum(f.result() for f in finished)
    dt = time.perf_counter() - t0
    # every chunk covers one p; the workload mixes the four p equally, which the
    # round-robin order reproduces up to the last partial round
    return done / dt, done, dt


def cpu_baseline(seconds: float, extra_modes: bool = True):
    """The oracle (as it stands) on the host cores: FP64 on every core (the
    reported value), and beside it FP64 on one core and the FP32 oracle on
    every core."""
    cores = os.cpu_count() or 1
    v, done, dt = _oracle_rate(seconds, cores, "f64")
    out = {"value": v, "unit": "shots/s", "cores": cores, "kind": "oracle",
           "sample": f"{done} depolarizing shots of the workload (X and Z decoded, p round-robin over "
                     f"{list(P_LIST)}), oracle FP64, {cores} threads (nproc {cores}), {dt:.1f} s"}
    if extra_modes:
        v1, d1, t1 = _oracle_rate(seconds / 3, 1, "f64")
        v32, d32, t32 = _oracle_rate(seconds / 3, cores, "f32")
        out["fp64_one_core"] = {"value": v1, "unit": "shots/s", "cores": 1, "sample": f"{d1} shots, {t1:.1f} s"}
        out["fp32_all_cores"] = {"value": v32, "unit": "shots/s", "cores": cores,
                                 "sample": f"{d32} shots, {t32:.1f} s"}
    return out


def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    budget = max(2.0, args.cpu_seconds / max(args.steps + args.warmup, 1))
    for _ in range(args.warmup):
        cpu_baseline(budget / 4, extra_modes=False)
    vals, t_all = [], time.perf_counter()
    for _ in range(args.steps):
        vals.append(cpu_baseline(budget, extra_modes=False)["value"])
    total = time.perf_counter() - t_all
    value = statistics.mean(vals)
    cb = cpu_baseline(budget, extra_modes=False)
    line = {
        "impl": "reference", "metric": "decoded shots/s", "value": value, "unit": "shots/s",
        "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": 1000 * total / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": WORKLOAD, "shots_per_p": args.shots},
        "cpu_baseline": {"value": value, "unit": "shots/s", "cores": cb["cores"], "kind": "oracle",
                         "sample": cb["sample"]},
        "e2e": {"value": value, "unit": "shots/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


MIXED = (("bb72", 8), ("bb144", 16), ("bb288", 32))
MIXED_P = 0.05


def mixed_measure(shots: int, steps: int, warmup: int, sample_clocks: bool = False):
    """[[72]], [[144]] and [[288]] shots 1:1:1 (R = 8 / 16 / 32), depolarizing
    p = 0.05, X and Z decoded: one autotuned, graph-captured mbbp_decode_mixed
    per step (a persistent launch per kernel body and small-code shape)
    against one plain mbbp_decode per (code, type) on the same syndromes
    (identical outputs, hence identical LER).  Returns the measurements."""
    import torch

    from paper_2605_14170_gb300 import mbbp
    from paper_2605_14170_gb300.inputs import named_code

    dev = torch.device("cuda", 0)
    torch.cuda.set_device(dev)
    per_code = max(1, shots // 3)
    entries = []  # (code, bases for X errors / Z errors, logicals)
    for name, R_ in MIXED:
        c = named_code(name)
        entries.append((c, mbbp.mbbp_build_bases(c.HZ, R_, SEED), mbbp.mbbp_build_bases(c.HX, R_, SEED + 1),
                        mbbp.mbbp_logicals_build(c.HZ, c.HX), mbbp.mbbp_logicals_build(c.HX, c.HZ)))
    bases = [b for e in entries for b in (e[1], e[2])]
    P = mbbp.mbbp_plan_create(bases)
    pm = 2 * MIXED_P / 3
    synd, llrs, errs = [], [], []
    for c, BZ, BX, _, _ in entries:
        n, W = c.n, (c.n + 31) // 32
        ex = torch.empty((per_code, W), dtype=torch.int32, device=dev)
        ez = torch.empty_like(ex)
        errs.append((ex, ez))
        l = torch.full((n,), float(np.log((1 - pm) / pm)), dtype=torch.float32, device=dev)
        for B in (BZ, BX):
            synd.append(torch.empty((per_code, B.m), dtype=torch.uint8, device=dev))
            llrs.append(l)
    ios, ws = mbbp.mixed_buffers(P, synd, llrs)

    def sample(k):
        for i, (c, BZ, BX, _, _) in enumerate(entries):
            ex, ez = errs[i]
            mbbp.mbbp_sample_errors(c.n, per_code, (k * 3 + i) * per_code, SEED, MIXED_P, mbbp.NOISE_DEPOLARIZING, ex, ez)
            mbbp.mbbp_syndrome(BZ, ex, synd[2 * i])
            mbbp.mbbp_syndrome(BX, ez, synd[2 * i + 1])

    sample(0)
    torch.cuda.synchronize()
    tuned_ms = mbbp.mbbp_plan_autotune(P, ios, ITERS, ALPHA, mbbp.RULE_NMS, ws)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        mbbp.mbbp_decode_mixed(P, ios, ITERS, ALPHA, mbbp.RULE_NMS, ws, stream=side)
        side.synchronize()
        with torch.cuda.graph(graph, stream=side):
            mbbp.mbbp_decode_mixed(P, ios, ITERS, ALPHA, mbbp.RULE_NMS, ws, stream=side)
    torch.cuda.current_stream().wait_stream(side)
    plain_out = [mbbp.decode(B, s, l, ITERS, ALPHA) for B, s, l in zip(bases, synd, llrs)]
    counts = torch.zeros((len(bases), 3), dtype=torch.int64, device=dev)
    launches = {"mixed": 0, "plain": 0}
    kinds = mbbp.mbbp_plan_info(P)["kind"]
    small = {entries[j // 2][0].name for j, k in enumerate(kinds) if k == 0}
    bp_launches = len(small) + (1 if any(k == 1 for k in kinds) else 0)
    dec_ms = {"mixed": [], "plain": []}

    def step_mixed(k, record):
        sample(k)
        if record:
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
        graph.replay()
        if record:
            e1.record()
            dec_ms["mixed"].append((e0, e1))
        for i, (_, _, _, LZ, LX) in enumerate(entries):
            mbbp.mbbp_judge(LZ, errs[i][0], ios[2 * i]["e_hat"], None, counts[2 * i])
            mbbp.mbbp_judge(LX, errs[i][1], ios[2 * i + 1]["e_hat"], None, counts[2 * i + 1])
        # sample+syndrome, BP (the generic launch and one per small-code shape;
        # each code here has its own shape), FWS per entry, judge
        launches["mixed"] = 9 + bp_launches + len(bases) + 6

    def step_plain(k, record):
        sample(k)
        if record:
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
        for j, (B, s, l) in enumerate(zip(bases, synd, llrs)):
            o = plain_out[j]
            mbbp.mbbp_decode(B, s, l, ITERS, ALPHA, mbbp.RULE_NMS, o["e_hat"], o["conv"], o["success"],
                             o["workspace"], iters_run=o["iters"], selected=o["selected"])
        if record:
            e1.record()
            dec_ms["plain"].append((e0, e1))
        launches["plain"] = 9 + 2 * len(bases)

    def timed(fn):
        for k in range(warmup):
            fn(k, False)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for k in range(steps):
            fn(warmup + k, True)
        e1.record()
        torch.cuda.synchronize()
        return e0.elapsed_time(e1)

    clk = ClockSampler(0) if sample_clocks else None
    if clk:
        clk.__enter__()
    ms_mixed = timed(step_mixed)
    if clk:
        clk.__exit__(None, None, None)
    counts_mixed = counts.clone()
    ms_plain = timed(step_plain)
    # identical outputs on the last step's syndromes
    same = all(torch.equal(x["e_hat"], o["e_hat"]) and torch.equal(x["iters"], o["iters"])
               for x, o in zip(ios, plain_out))
    n_shots = steps * 3 * per_code
    info = mbbp.mbbp_plan_info(P)
    cnt = counts_mixed.cpu().numpy()
    names = [f"{c.name}:{t}" for c, *_ in entries for t in ("X", "Z")]
    dm = statistics.mean(a.elapsed_time(b) for a, b in dec_ms["mixed"])
    dp = statistics.mean(a.elapsed_time(b) for a, b in dec_ms["plain"])
    return {
        "shots_per_step": 3 * per_code, "steps": steps, "warmup": warmup,
        "value": n_shots / (ms_mixed / 1e3), "unit": "shots/s", "ms_per_step": ms_mixed / steps,
        "decode_ms": dm,
        "plain": {"value": n_shots / (ms_plain / 1e3), "unit": "shots/s", "ms_per_step": ms_plain / steps,
                  "decode_ms": dp, "launches_per_step": launches["plain"]},
        "speedup_vs_plain": ms_plain / ms_mixed, "decode_speedup_vs_plain": dp / dm,
        "outputs_identical_to_plain": bool(same),
        "ler": {nm: float(cnt[j, 1] + cnt[j, 2]) / (steps * per_code) for j, nm in enumerate(names)},
        "plan": {"warps": info["warps"], "chunk": info["chunk"], "kind": info["kind"], "order": info["order"],
                 "autotuned_ms": tuned_ms},
        "launches_per_step": launches["mixed"],
        "clocks": clk.summary() if clk else None,
    }


MIXED_WORKLOAD = ("mixed batch: [[72,12,6]] R=8, [[144,12,12]] R=16, [[288,12,18]] R=32, 1:1:1, depolarizing "
                  "p=0.05, X and Z decoded, 100 iters, persistent autotuned launches (one per kernel body and "
                  "small-code shape) replayed as one CUDA graph")


def run_mixed(args):
    """The mixed-batch workload as its own JSON line."""
    r = mixed_measure(args.shots, args.steps, args.warmup, sample_clocks=True)
    line = {
        "metric": "decoded shots/s", "value": r["value"], "unit": "shots/s", "n_gpus": 1,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": r["ms_per_step"],
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": MIXED_WORKLOAD, "shots_per_step": r["shots_per_step"], "alpha": ALPHA},
        "plain": r["plain"], "speedup_vs_plain": r["speedup_vs_plain"],
        "decode_speedup_vs_plain": r["decode_speedup_vs_plain"],
        "outputs_identical_to_plain": r["outputs_identical_to_plain"], "ler": r["ler"], "plan": r["plan"],
        "gpu_launches": r["launches_per_step"] * args.steps, "clocks": r["clocks"],
    }
    print(json.dumps(line), flush=True)


GB882_P = (0.02, 0.03, 0.04, 0.05, 0.06)


def gb882_measure(shots: int, steps: int = 1, warmup: int = 1, p_list=None, wms: bool = False):
    """Plain MBBP-LD on the length-882 GB code (R = 64, 100 iterations,
    depolarizing p in {0.02 .. 0.06}, X errors decoded with H_Z): shots/s per
    p from CUDA events around each decode call (BP + FWS), inputs resident.
    With `wms`, also the learned-form decoder (mbbp_wms_decode, T = 25) with
    its initial weights w = alpha, g = 0, which decide exactly as plain
    MBBP-LD: the same work through the weighted kernel."""
    import torch

    from paper_2605_14170_gb300 import mbbp
    from paper_2605_14170_gb300.inputs import named_code

    dev = torch.device("cuda", 0)
    c = named_code("gb882")
    n, W = c.n, (c.n + 31) // 32
    t0 = time.perf_counter()
    B = mbbp.mbbp_build_bases(c.HZ, 64, SEED)
    build_s = time.perf_counter() - t0
    ex = torch.empty((shots, W), dtype=torch.int32, device=dev)
    ez = torch.empty_like(ex)
    syn = torch.empty((shots, B.m), dtype=torch.uint8, device=dev)
    out = None
    per_p = {}
    p_list = GB882_P if p_list is None else p_list
    for ip, p in enumerate(p_list):
        mbbp.mbbp_sample_errors(n, shots, 90_000_000_000 + ip * shots, SEED, p, mbbp.NOISE_DEPOLARIZING, ex, ez)
        mbbp.mbbp_syndrome(B, ex, syn)
        pm = 2 * p / 3
        llr = torch.full((n,), float(np.log((1 - pm) / pm)), dtype=torch.float32, device=dev)
        if out is None:
            out = mbbp.decode(B, syn, llr, ITERS, ALPHA)
        times = []
        for k in range(warmup + steps):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            mbbp.mbbp_decode(B, syn, llr, ITERS, ALPHA, mbbp.RULE_NMS, out["e_hat"], out["conv"], out["success"],
                             out["workspace"], iters_run=out["iters"], selected=out["selected"])
            e1.record()
            e1.synchronize()
            if k >= warmup:
                times.append(e0.elapsed_time(e1))
        ms = statistics.mean(times)
        it = (out["iters"].to(torch.int64) & 0xFFFF).float().mean().item()
        per_p[str(p)] = {"shots_per_s": shots / (ms / 1e3), "decode_ms": ms, "mean_K": it,
                         "success": float(out["success"].float().mean().item())}
        if wms:
            w, g = mbbp.wms_params(B, 25, alpha=ALPHA, device=dev)
            o2 = {k: torch.empty_like(v) for k, v in out.items()}
            o2["workspace"] = torch.empty(mbbp.mbbp_wms_decode_workspace_size(B, shots, 25), dtype=torch.uint8,
                                          device=dev)
            wt = []
            for k in range(warmup + steps):
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record()
                mbbp.mbbp_wms_decode(B, syn, llr, ITERS, 25, w, g, o2["e_hat"], o2["conv"], o2["success"],
                                     o2["workspace"], iters_run=o2["iters"], selected=o2["selected"])
                e1.record()
                e1.synchronize()
                if k >= warmup:
                    wt.append(e0.elapsed_time(e1))
            wms_ms = statistics.mean(wt)
            per_p[str(p)]["wms_decode_ms"] = wms_ms
            per_p[str(p)]["wms_shots_per_s"] = shots / (wms_ms / 1e3)
            per_p[str(p)]["wms_identical_to_plain"] = bool(torch.equal(o2["e_hat"], out["e_hat"]))
    total_ms = sum(v["decode_ms"] for v in per_p.values())
    return {"workload": "length-882 GB code (seeded, k=4), R=64, 100 iters, alpha 0.625, flooding, FWS, "
                        "depolarizing X errors", "shots_per_p": shots, "steps": steps, "warmup": warmup,
            "shots_per_s": len(p_list) * shots / (total_ms / 1e3), "per_p": per_p,
            "bases_build_s": build_s}


def run_gb882(args):
    """Plain MBBP-LD on the length-882 GB code as its own JSON line (`--p`
    picks one p; default all five)."""
    r = gb882_measure(args.shots, args.steps, args.warmup, None if args.p is None else (args.p,), wms=args.wms)
    ms = sum(v["decode_ms"] for v in r["per_p"].values())
    line = {"metric": "decoded shots/s", "value": r["shots_per_s"], "unit": "shots/s", "n_gpus": 1,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": r["workload"], "shots_per_p": args.shots}, "per_p": r["per_p"]}
    print(json.dumps(line), flush=True)


def run_learned(args):
    """Learned-weight vs plain MBBP-LD on the length-882 GB code (R = 64,
    100 iterations, depolarizing p in {0.02 .. 0.06}, X errors): WMS trained
    on the GPU by the library's kernels (T = 25, checkpoint every 5,
    validation-selected), then both decoders on the same fresh shots."""
    import time as _time

    import torch

    from paper_2605_14170_gb300 import learn, mbbp
    from paper_2605_14170_gb300.inputs import named_code

    dev = torch.device("cuda", 0)
    torch.cuda.set_device(dev)
    c = named_code("gb882")
    B = mbbp.mbbp_build_bases(c.HZ, 64, SEED)
    L = mbbp.mbbp_logicals_build(c.HZ, c.HX)
    t0 = _time.time()
    # trained at p = 0.07 and selected on held-out shots at p = 0.08, where the
    # code fails often enough to tell weights apart (below 0.06 its LER is
    # under 1e-4 and 1e4 held-out shots show no failure for any weights)
    # the best trained weights on the held-out shots (the initial weights are
    # left out of the choice, so the comparison below is of trained weights)
    w, g, hist = learn.train_wms(B, 0.07, T=25, ckpt=5, batch=args.train_batch, steps=args.train_steps,
                                 lr=1e-3, L=L, val_shots=20000, val_every=25, log_every=0, val_p=0.08,
                                 keep_initial=False)
    torch.cuda.synchronize()
    train_s = _time.time() - t0
    shots = args.shots
    res = {}
    for p in (0.02, 0.03, 0.04, 0.05, 0.06, 0.07, 0.08):
        # 10x the shots where plain MBBP-LD fails often enough to resolve a difference
        res[str(p)] = learn.compare_ler(B, L, w, g, p, shots * (10 if p >= 0.06 else 1), ITERS, chunk=100000)
    # throughput of the two decoders on one batch of p = 0.04 syndromes
    n, W = c.n, (c.n + 31) // 32
    ex = torch.empty((shots, W), dtype=torch.int32, device=dev)
    ez = torch.empty_like(ex)
    mbbp.mbbp_sample_errors(n, shots, 77_000_000_000, SEED, 0.04, mbbp.NOISE_DEPOLARIZING, ex, ez)
    syn = torch.empty((shots, B.m), dtype=torch.uint8, device=dev)
    mbbp.mbbp_syndrome(B, ex, syn)
    pm = 2 * 0.04 / 3
    llr = torch.full((n,), float(np.log((1 - pm) / pm)), dtype=torch.float32, device=dev)

    def timed(fn):
        for _ in range(args.warmup):
            fn()
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(args.steps):
            fn()
        e1.record()
        torch.cuda.synchronize()
        return e0.elapsed_time(e1) / args.steps

    ms_plain = timed(lambda: mbbp.decode(B, syn, llr, ITERS, ALPHA))
    ms_learned = timed(lambda: mbbp.wms_decode(B, syn, llr, ITERS, w, g))
    # the same recipe on [[144,12,12]] with R = 8, where the LER is high
    # enough for the weights to make a measurable difference
    c2 = named_code("bb144")
    B2 = mbbp.mbbp_build_bases(c2.HZ, 8, SEED)
    L2 = mbbp.mbbp_logicals_build(c2.HZ, c2.HX)
    w2, g2, hist2 = learn.train_wms(B2, 0.05, T=25, ckpt=5, batch=2048, steps=150, lr=1e-3, L=L2,
                                    val_shots=30000, val_every=25, log_every=0)
    res2 = {str(pp): learn.compare_ler(B2, L2, w2, g2, pp, 200_000, ITERS) for pp in (0.03, 0.04, 0.05, 0.06)}
    line = {
        "metric": "decoded shots/s", "value": shots / (ms_learned / 1e3), "unit": "shots/s", "n_gpus": 1,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_learned, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": "learned-weight vs plain MBBP-LD, length-882 GB code (seeded, k=4), R=64, "
                               "100 iters, depolarizing X errors; WMS T=25, checkpoint 5, trained on GPU at "
                               "p=0.07, the best trained weights on held-out shots at p=0.08; 1e6 shots per p "
                               "for p >= 0.06",
                   "shots_per_p": shots, "train_batch": args.train_batch, "train_steps": args.train_steps},
        "plain": {"value": shots / (ms_plain / 1e3), "unit": "shots/s", "ms_per_step": ms_plain},
        "train_s": train_s,
        "selected_step": min((h for h in hist if h[0] > 0),
                             key=lambda h: (h[2] if h[2] is not None else 1 << 60))[0],
        "validation_failures": {str(h[0]): h[2] for h in hist if h[2] is not None},
        "ler": {p: {"plain": r["plain"]["ler"], "plain_ci95": r["plain"]["ci95"],
                    "learned": r["learned"]["ler"], "learned_ci95": r["learned"]["ci95"],
                    "plain_failures": r["plain"]["failures"], "learned_failures": r["learned"]["failures"],
                    "shots": r["shots"],
                    "z_plain_minus_learned": learn.two_proportion_z(r["plain"]["failures"], r["learned"]["failures"],
                                                                    r["shots"])}
                for p, r in res.items()},
        "bb144_r8": {"train": "150 steps x 2048 shots at p=0.05, validation-selected",
                     "selected_step": min(hist2, key=lambda h: (h[2] if h[2] is not None else 1 << 60))[0],
                     "ler": {p: {"plain_failures": r["plain"]["failures"], "learned_failures": r["learned"]["failures"],
                                 "shots": r["shots"], "plain_ci95": r["plain"]["ci95"],
                                 "learned_ci95": r["learned"]["ci95"]} for p, r in res2.items()}},
    }
    print(json.dumps(line), flush=True)


def run_paper(args):
    """The paper's own decoder setting on [[288,12,18]] (Section IV: binary
    symmetric channel of independent X errors at p_x in {0.04, 0.06, 0.08},
    serial schedule, alpha = 0.875, 100 iterations; R = 20 subtree
    representations, the partition count of Table II).  On the same shots: FWS (the paper's
    rule) and LMS (classical MBBP), the matched random augmentation of
    Table II, and flooding at alpha = 0.625.  ``value`` = shots/s of the
    serial FWS decoder; per decoder: LER with its 95% interval, mean
    iterations and shots/s."""
    import torch

    from paper_2605_14170_gb300 import learn, mbbp
    from paper_2605_14170_gb300.inputs import named_code

    dev = torch.device("cuda", 0)
    torch.cuda.set_device(dev)
    c = named_code("bb288")
    H = c.HZ
    m, n = H.shape
    Rp = 20
    B = mbbp.mbbp_build_bases(H, Rp, SEED)
    sizes = [len(x) for x in B.sets]
    Br = mbbp.mbbp_build_bases_from_sets(H, mbbp.mbbp_random_sets(m, sizes, SEED + 7))
    L = mbbp.mbbp_logicals_build(H, c.HX)
    S = args.shots
    W = (n + 31) // 32
    ex = torch.empty((S, W), dtype=torch.int32, device=dev)
    syn = torch.empty((S, m), dtype=torch.uint8, device=dev)
    decoders = {
        "serial_fws": (B, 0.875, mbbp.SCHEDULE_SERIAL, mbbp.DECISION_FWS),
        "serial_lms": (B, 0.875, mbbp.SCHEDULE_SERIAL, mbbp.DECISION_LMS),
        "serial_fws_random_sets": (Br, 0.875, mbbp.SCHEDULE_SERIAL, mbbp.DECISION_FWS),
        "flooding_fws_alpha0.625": (B, 0.625, mbbp.SCHEDULE_FLOODING, mbbp.DECISION_FWS),
    }
    edges = {k: torch.from_numpy(d[0].edges.astype(np.int64)).to(dev) for k, d in decoders.items()}
    res = {k: {} for k in decoders}
    tot_ms = {k: 0.0 for k in decoders}
    tot_shots = 0
    tot_work = {k: 0 for k in decoders}
    ncalls = 0
    with ClockSampler(0) as clk:
        for ip, p in enumerate((0.04, 0.06, 0.08)):
            llr = torch.full((n,), float(np.log((1 - p) / p)), dtype=torch.float32, device=dev)
            fails = {k: torch.zeros(3, dtype=torch.int64, device=dev) for k in decoders}
            iters_sum = {k: 0.0 for k in decoders}
            for k in range(args.warmup + args.steps):
                mbbp.mbbp_sample_errors(n, S, (ip * 1000 + k) * S, SEED, p, mbbp.NOISE_BSC, ex, None)
                mbbp.mbbp_syndrome(B, ex, syn)
                for name, (BB, alpha, sch, dec) in decoders.items():
                    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                    e0.record()
                    out = mbbp.decode(BB, syn, llr, ITERS, alpha, schedule=sch, decision=dec)
                    e1.record()
                    if k < args.warmup:
                        continue
                    mbbp.mbbp_judge(L, ex, out["e_hat"], None, fails[name])
                    it = out["iters"].to(torch.int64) & 0xFFFF
                    torch.cuda.synchronize()
                    tot_ms[name] += e0.elapsed_time(e1)
                    iters_sum[name] += float(it.float().mean().item())
                    tot_work[name] += int((it.sum(0) * edges[name]).sum().item())
                    ncalls += 1 if name == "serial_fws" else 0
                if k >= args.warmup:
                    tot_shots += S
            for name in decoders:
                f = fails[name].cpu().numpy()
                kf = int(f[1] + f[2])
                res[name][str(p)] = {"failures": kf, "ler": kf / (args.steps * S),
                                     "ci95": learn.wilson(kf, args.steps * S),
                                     "mean_iters": iters_sum[name] / args.steps}
    shots_per_decoder = tot_shots
    line = {
        "metric": "decoded shots/s", "value": shots_per_decoder / (tot_ms["serial_fws"] / 1e3),
        "unit": "shots/s", "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": tot_ms["serial_fws"] / (3 * args.steps), "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": "paper setting: [[288,12,18]] BB, independent X errors (BSC) at p_x in "
                               "{0.04,0.06,0.08}, R=20 subtree representations, serial schedule, "
                               "alpha=0.875, 100 iters, FWS", "shots_per_p_per_step": S},
        "decoders": {name: {"shots_per_s": shots_per_decoder / (tot_ms[name] / 1e3),
                            "edge_updates_per_s": tot_work[name] / (tot_ms[name] / 1e3),
                            "ler": res[name]} for name in decoders},
        "random_set_sizes": sizes,
        "gpu_launches": 3 * args.steps * (2 + 2 * len(decoders)),
        "clocks": clk.summary(),
    }
    print(json.dumps(line), flush=True)


def wms_measure(steps: int, warmup: int, sample_clocks: bool = False):
    """One training step of differentiable weighted min-sum per bench step on
    [[144,12,12]] (R = 8 subtree representations, T = 25 unrolled flooding
    iterations, per-edge per-iteration weights and damping, checkpoint
    every 5 iterations, batch 4096 depolarizing X errors at p = 0.06, BCE of
    every iteration's posterior): sample + syndrome + forward + hand-written
    adjoint + two Adam steps, all in the library's kernels.  ``value`` =
    training syndromes/s; the forward and backward kernels are timed
    separately with CUDA events."""
    import torch

    from paper_2605_14170_gb300 import mbbp
    from paper_2605_14170_gb300.inputs import named_code

    dev = torch.device("cuda", 0)
    torch.cuda.set_device(dev)
    c = named_code("bb144")
    B = mbbp.mbbp_build_bases(c.HZ, 8, SEED)
    T, ckpt, batch, p = 25, 5, 4096, 0.06
    n, W = c.n, (c.n + 31) // 32
    w, g = mbbp.wms_params(B, T, alpha=ALPHA, device=dev)
    mw, vw, mg, vg = (torch.zeros_like(w) for _ in range(4))
    gw, gg = torch.zeros_like(w), torch.zeros_like(g)
    ex = torch.empty((batch, W), dtype=torch.int32, device=dev)
    ez = torch.empty_like(ex)
    syn = torch.empty((batch, B.m), dtype=torch.uint8, device=dev)
    post = torch.empty((batch, B.R, n), dtype=torch.float32, device=dev)
    loss = torch.empty((batch, B.R), dtype=torch.float32, device=dev)
    ws_bytes = mbbp.mbbp_wms_workspace_size(B, batch, T, ckpt)
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device=dev)
    pm = 2 * p / 3
    llr = torch.full((n,), float(np.log((1 - pm) / pm)), dtype=torch.float32, device=dev)
    scale = 1.0 / (batch * B.R * n)
    ev = []

    def step(k, record):
        mbbp.mbbp_sample_errors(n, batch, k * batch, SEED, p, mbbp.NOISE_DEPOLARIZING, ex, ez)
        mbbp.mbbp_syndrome(B, ex, syn)
        e = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
        e[0].record()
        mbbp.mbbp_wms_forward(B, syn, llr, T, w, g, ckpt, ex, scale, post, loss, ws, all_iters=True)
        e[1].record()
        gw.zero_()
        gg.zero_()
        mbbp.mbbp_wms_backward(B, syn, llr, T, w, g, ckpt, ex, scale, post, gw, gg, ws, all_iters=True)
        e[2].record()
        mbbp.mbbp_adam_step(w, gw, mw, vw, 1e-3, 0.9, 0.999, 1e-8, k + 1, 0.0, 2.0)
        mbbp.mbbp_adam_step(g, gg, mg, vg, 1e-3, 0.9, 0.999, 1e-8, k + 1, 0.0, 0.9)
        if record:
            ev.append(e)

    for k in range(warmup):
        step(k, False)
    torch.cuda.synchronize()
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    clk = ClockSampler(0) if sample_clocks else None
    if clk:
        clk.__enter__()
    t0.record()
    for k in range(steps):
        step(warmup + k, True)
    t1.record()
    torch.cuda.synchronize()
    if clk:
        clk.__exit__(None, None, None)
    ms = t0.elapsed_time(t1)
    fwd = statistics.mean(a.elapsed_time(b) for a, b, _ in ev)
    bwd = statistics.mean(b.elapsed_time(c_) for _, b, c_ in ev)
    E = int(B.edges.sum())
    upd = batch * T * E  # forward message updates per step (every edge of every representation)
    ck_bytes = batch * B.R * int(B.edges.max()) * 4 * ((T - 1) // ckpt)
    full_bytes = batch * B.R * int(B.edges.max()) * 4 * T
    return {
        "metric": "training syndromes/s", "value": steps * batch / (ms / 1e3), "unit": "syndromes/s",
        "n_gpus": 1, "steps": steps, "warmup": warmup, "ms_per_step": ms / steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": "weighted min-sum training step: [[144,12,12]] R=8, T=25 unrolled iterations, "
                               "per-edge per-iteration weights + damping, checkpoint every 5, batch 4096, "
                               "depolarizing p=0.06, BCE of every iteration", "batch": batch, "T": T, "ckpt": ckpt},
        "forward_ms": fwd, "backward_ms": bwd,
        "forward_edge_updates_per_s": upd / (fwd / 1e3),
        "workspace_bytes": ws_bytes, "message_bytes_checkpointed": ck_bytes,
        "message_bytes_without_checkpoints": full_bytes,
        "loss": float(loss.sum().item()),
        "gpu_launches": steps * 8,
        "clocks": clk.summary() if clk else None,
    }


def run_wms(args):
    """The weighted min-sum training step as its own JSON line."""
    print(json.dumps(wms_measure(args.steps, args.warmup, sample_clocks=True)), flush=True)


def bb72_measure(reps: int = 20):
    """The small configuration: [[72,12,6]], X errors (BSC) p = 0.05 decoded
    with H_Z, R = 4, 50 iterations, alpha = 0.625, 2000 seeded shots; the
    decode call (BP + FWS) timed with CUDA events, averaged over `reps`
    calls on the same syndromes (a 2000-shot launch is latency-bound)."""
    import torch

    from paper_2605_14170_gb300 import mbbp
    from paper_2605_14170_gb300.inputs import named_code

    dev = torch.device("cuda", 0)
    c = named_code("bb72")
    shots, n = 2000, c.n
    B = mbbp.mbbp_build_bases(c.HZ, 4, 20260514)
    L = mbbp.mbbp_logicals_build(c.HZ, c.HX)
    W = (n + 31) // 32
    ex = torch.empty((shots, W), dtype=torch.int32, device=dev)
    mbbp.mbbp_sample_errors(n, shots, 0, 20260514, 0.05, mbbp.NOISE_BSC, ex)
    syn = torch.empty((shots, B.m), dtype=torch.uint8, device=dev)
    mbbp.mbbp_syndrome(B, ex, syn)
    llr = torch.full((n,), float(np.log(0.95 / 0.05)), dtype=torch.float32, device=dev)
    out = mbbp.decode(B, syn, llr, 50, ALPHA)
    times = []
    for _ in range(reps + 3):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        mbbp.mbbp_decode(B, syn, llr, 50, ALPHA, mbbp.RULE_NMS, out["e_hat"], out["conv"], out["success"],
                         out["workspace"], iters_run=out["iters"], selected=out["selected"])
        e1.record()
        e1.synchronize()
        times.append(e0.elapsed_time(e1))
    ms = statistics.mean(times[3:])
    cnt = torch.zeros(3, dtype=torch.int64, device=dev)
    mbbp.mbbp_judge(L, ex, out["e_hat"], None, cnt)
    c3 = cnt.cpu().numpy()
    return {"workload": "[[72,12,6]] BB, X errors (BSC) p=0.05 decoded with H_Z, R=4, 50 iters, alpha 0.625, "
                        "2000 shots", "decode_ms": ms, "shots_per_s": shots / (ms / 1e3),
            "failures": int(c3[1] + c3[2]), "shots": shots}


def main():
    args = parse()
    if args.shots is None:
        args.shots = {"mixed": 300_000, "learned": 100_000, "paper": 200_000, "gb882": 100_000}.get(args.workload,
                                                                                                   1_000_000)
    if args.impl == "reference":
        run_reference(args)
        return
    if args.workload == "mixed":
        run_mixed(args)
        return
    if args.workload == "learned":
        run_learned(args)
        return
    if args.workload == "paper":
        run_paper(args)
        return
    if args.workload == "wms":
        run_wms(args)
        return
    if args.workload == "gb882":
        run_gb882(args)
        return

    import torch
    import torch.distributed as dist

    from paper_2605_14170_gb300 import mbbp, shard
    from paper_2605_14170_gb300.inputs import named_code

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        dist.init_process_group("nccl")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    stream = torch.cuda.current_stream()

    code = named_code(CODE)
    n = code.n
    W = (n + 31) // 32
    S = args.shots
    t_build = time.perf_counter()
    BZ = mbbp.mbbp_build_bases(code.HZ, R, SEED)       # X errors
    BX = mbbp.mbbp_build_bases(code.HX, R, SEED + 1)   # Z errors
    t_build = time.perf_counter() - t_build
    LZ = mbbp.mbbp_logicals_build(code.HZ, code.HX)
    LX = mbbp.mbbp_logicals_build(code.HX, code.HZ)
    m = code.HZ.shape[0]
    llrs = {p: torch.full((n,), float(np.log((1 - 2 * p / 3) / (2 * p / 3))), dtype=torch.float32, device=dev)
            for p in P_LIST}
    edges = {"Z": torch.from_numpy(BZ.edges.astype(np.int64)).to(dev),
             "X": torch.from_numpy(BX.edges.astype(np.int64)).to(dev)}

    ex = torch.empty((S, W), dtype=torch.int32, device=dev)
    ez = torch.empty((S, W), dtype=torch.int32, device=dev)
    syn = torch.empty((S, m), dtype=torch.uint8, device=dev)
    ws = torch.empty(mbbp.mbbp_decode_workspace_size(BZ, S), dtype=torch.uint8, device=dev)
    e_hat = torch.empty((S, n), dtype=torch.uint8, device=dev)
    conv = torch.empty((S, R), dtype=torch.uint8, device=dev)
    iters = torch.empty((S, R), dtype=torch.int16, device=dev)
    succ = torch.empty((S,), dtype=torch.uint8, device=dev)
    fail_x = torch.empty((S,), dtype=torch.uint8, device=dev)
    fail_z = torch.empty((S,), dtype=torch.uint8, device=dev)
    counts = torch.zeros((len(P_LIST), 3, 3), dtype=torch.int64, device=dev)  # p, type(X,Z,any), code
    work = torch.zeros((), dtype=torch.int64, device=dev)
    # per p: sum over (shot, representation) of K, and sum over shots of the
    # largest K of the shot's representations (the latency term), X and Z
    kstats = torch.zeros((len(P_LIST), 2), dtype=torch.int64, device=dev)
    dec_events = []
    launches_per_step = 0

    # Every decode call (one p, one error type: counter reset, persistent BP
    # kernel, FWS) is captured once into a CUDA graph and replayed each step;
    # its inputs and outputs stay in the same buffers.  One direct call per
    # graph first sets the kernels' shared-memory limits and occupancy.
    syn.zero_()
    side = torch.cuda.Stream()
    side.wait_stream(stream)
    graphs = {}
    with torch.cuda.stream(side):
        for p in P_LIST:
            for key, B in (("Z", BZ), ("X", BX)):
                def call(B=B, p=p):
                    mbbp.mbbp_decode(B, syn, llrs[p], ITERS, ALPHA, mbbp.RULE_NMS, e_hat, conv, succ, ws,
                                     iters_run=iters, stream=side)
                call()
                side.synchronize()
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g, stream=side):
                    call()
                graphs[(p, key)] = g
    stream.wait_stream(side)
    torch.cuda.synchronize()

    def step(k, record=False):
        nonlocal launches_per_step
        launches = 0
        for ip, p in enumerate(P_LIST):
            first = shard.first_shot(k, rank, world, ip, len(P_LIST), S)
            mbbp.mbbp_sample_errors(n, S, first, SEED, p, mbbp.NOISE_DEPOLARIZING, ex, ez)
            launches += 1
            for key, B, L, e, fl in (("Z", BZ, LZ, ex, fail_x), ("X", BX, LX, ez, fail_z)):
                mbbp.mbbp_syndrome(B, e, syn)
                if record:
                    ev0 = torch.cuda.Event(enable_timing=True)
                    ev1 = torch.cuda.Event(enable_timing=True)
                    ev0.record(stream)
                graphs[(p, key)].replay()
                if record:
                    ev1.record(stream)
                    dec_events.append((ev0, ev1, key))
                mbbp.mbbp_judge(L, e, e_hat, fl, counts[ip, 0 if key == "Z" else 1])
                launches += 4  # syndrome, BP, FWS, judge
                it64 = iters.to(torch.int64) & 0xFFFF
                work.add_((it64.sum(0) * edges[key]).sum())
                kstats[ip, 0] += it64.sum()
                kstats[ip, 1] += it64.max(1).values.sum()
            # any-type failure for the combined logical error rate
            counts[ip, 2, 1] += ((fail_x != 0) | (fail_z != 0)).sum()
        launches_per_step = launches

    for k in range(args.warmup):
        step(k)
    torch.cuda.synchronize()
    counts.zero_()
    work.zero_()
    kstats.zero_()
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    t0 = torch.cuda.Event(enable_timing=True)
    t1 = torch.cuda.Event(enable_timing=True)
    with ClockSampler(local) as clk:
        t0.record(stream)
        for k in range(args.steps):
            step(args.warmup + k, record=True)
        t1.record(stream)
        torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    ms = shard.max_over_ranks(dist, t0.elapsed_time(t1), dev)
    shard.reduce_counters(dist, counts, work, kstats)
    shots_total = args.steps * len(P_LIST) * S * world
    value = shots_total / (ms / 1000.0)
    edge_updates = int(work.item())
    dec_ms = [a.elapsed_time(b) for a, b, _ in dec_events]
    dec_avg_ms = statistics.mean(dec_ms)
    # per-launch algorithmic work of the decode call
    edge_per_launch = edge_updates / max(len(dec_ms) * world, 1)
    peaks, peak_kind = read_peaks()
    props = torch.cuda.get_device_properties(dev)
    sm_count = props.multi_processor_count
    f_max = peaks.get("sm_max_mhz", 2070.0) * 1e6
    peak_ops = sm_count * OPS_PER_EDGE_UPDATE * EDGE_UPDATES_PER_CLK_SM * f_max
    peak_ops_128 = sm_count * 128 * f_max  # every operation at the fma pipe's 128 lanes
    achieved_ops = OPS_PER_EDGE_UPDATE * edge_per_launch / (dec_avg_ms / 1000.0)
    cnt = counts.cpu().numpy()
    ks = kstats.cpu().numpy()
    ler = {str(p): {"x": float(cnt[i, 0, 2] + cnt[i, 0, 1]) / (args.steps * S * world),
                    "z": float(cnt[i, 1, 2] + cnt[i, 1, 1]) / (args.steps * S * world),
                    "any": float(cnt[i, 2, 1]) / (args.steps * S * world)} for i, p in enumerate(P_LIST)}

    e2e = None
    if not args.no_e2e:
        e2e = run_e2e(args, mbbp, BZ, BX, llrs, S, dev, stream, rank, world)

    extra = None
    if rank == 0 and world == 1 and not args.no_extra:
        # the other configurations, measured on the same GPU after the
        # headline's timed region: the mixed batch (3e5 shots, graph-replayed
        # persistent launches vs per-code launches), plain MBBP-LD on the
        # length-882 GB code with R = 64, the weighted min-sum training step
        # and the small [[72,12,6]] decode
        extra = {"mixed": mixed_measure(300_000, 5, 3), "gb882_r64_plain": gb882_measure(100_000),
                 "wms_training": wms_measure(5, 3), "bb72_r4": bb72_measure()}
        extra["mixed"]["workload"] = MIXED_WORKLOAD

    cb = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        cb = cpu_baseline(args.cpu_seconds)
    clocks = clk.summary()
    probe = measure_probes(mbbp, stream, sm_count, clocks.get("sm_mhz") or peaks.get("sm_max_mhz", 2070.0))

    if rank == 0:
        line = {
            "metric": "decoded shots/s", "value": value, "unit": "shots/s", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic",
            "config": {"workload": WORKLOAD, "code": "[[144,12,12]]", "R": R, "iters": ITERS,
                       "alpha": ALPHA, "rule": "normalized min-sum, flooding", "p": list(P_LIST),
                       "shots_per_p_per_gpu": S, "noise": "code-capacity depolarizing",
                       "launch": "each decode call (persistent BP kernel + FWS) captured once as a CUDA "
                                 "graph and replayed every step; sampling, syndrome and judge launched directly",
                       "l2": "inputs larger than L2 (per decode call: "
                             f"{S * m / 1e6:.0f} MB syndromes, {ws.numel() / 1e6:.0f} MB workspace, "
                             f"{S * n / 1e6:.0f} MB estimates)"},
            "bases_build_s": t_build,
            "edge_updates_per_s": edge_updates / (ms / 1000.0),
            "edge_updates_per_shot": edge_updates / shots_total,
            "edge_updates_per_shot_dense_bound": 2 * R * float(np.mean(BZ.edges)) * ITERS,
            "decoded_syndromes_per_s": 2 * value,
            "iterations": {str(p): {"mean_K": float(ks[i, 0]) / (2 * args.steps * S * world * R),
                                    "mean_K_max_per_shot": float(ks[i, 1]) / (2 * args.steps * S * world)}
                           for i, p in enumerate(P_LIST)},
            "ler": ler,
            "roofline": {"bound": "alu", "achieved": achieved_ops / 1e12, "peak": peak_ops_128 / 1e12,
                         "unit": "Tops/s", "frac": achieved_ops / peak_ops_128,
                         "traffic": DRAM_BYTES_PER_SHOT * S if DRAM_BYTES_PER_SHOT is not None else None,
                         "traffic_note": "dram read+write of the BP kernel from one ncu capture of a "
                                         "100k-shot launch of the current kernel "
                                         "(profiles/kernels_current.md), scaled by shots",
                         "kernel": "mbbp_decode (BP + FWS)", "decode_ms_avg": dec_avg_ms,
                         "edge_updates_per_launch": edge_per_launch,
                         "ops_per_edge_update": OPS_PER_EDGE_UPDATE,
                         "peak_basis": f"{sm_count} SMs x 128 lanes x {peaks.get('sm_max_mhz', 2070.0)} MHz "
                                       f"({peak_kind} max SM clock): every algorithmic operation at one lane-issue",
                         "peak_op_mix": peak_ops / 1e12, "frac_op_mix": achieved_ops / peak_ops,
                         "peak_op_mix_basis": f"{sm_count} SMs x {peaks.get('sm_max_mhz', 2070.0)} MHz x "
                                              f"{OPS_PER_EDGE_UPDATE} ops x min({ALU_LANES}/{ALU_OPS} alu, "
                                              f"{FMA_LANES}/{FMA_OPS} fma, {ISSUE_LANES}/{OPS_PER_EDGE_UPDATE} "
                                              "issue) edge-updates per SM per clock; pipe widths confirmed by "
                                              "the probes",
                         "probe": probe},
            "gpu_launches": launches_per_step * args.steps,
            "clocks": clocks,
        }
        if e2e is not None:
            line["e2e"] = e2e
        if extra is not None:
            line["extra"] = extra
        if cb is not None:
            line["cpu_baseline"] = cb
        print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()


def measure_probes(mbbp, stream, sm_count, mhz):
    """Per-SM rates of the throughput probes (FP32 add, FP32 min/max, 3-input
    logic: lanes per clock; 16-byte shared-memory loads: bytes per clock), the
    best of three launches each, at the SM clock sampled during the timed
    region."""
    import torch
    sink = torch.zeros(1, dtype=torch.float32, device=stream.device)
    out = {}
    for kind, name in ((mbbp.PROBE_FADD, "fadd_lanes"), (mbbp.PROBE_FMNMX, "fmnmx_lanes"),
                       (mbbp.PROBE_LOP3, "lop3_lanes"), (mbbp.PROBE_SMEM, "smem_bytes")):
        mbbp.mbbp_probe(kind, 64, sink, stream=stream)
        best = 0.0
        for _ in range(3):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            work = mbbp.mbbp_probe(kind, 2048, sink, stream=stream)
            e1.record(stream)
            e1.synchronize()
            best = max(best, work / (e0.elapsed_time(e1) * 1e-3) / sm_count / (mhz * 1e6))
        out[name + "_per_clk_per_sm"] = round(best, 2)
    out["sm_mhz"] = mhz
    return out


def run_e2e(args, mbbp, BZ, BX, llrs, S, dev, stream, rank, world):
    """Same metric through mbbp_decode with host buffers: pinned syndromes in,
    estimates / flags / success out, inside the timed region (copies
    double-buffered on two copy streams, overlapping the decodes)."""
    import torch
    n, m = BZ.n, BZ.m
    W = (n + 31) // 32
    # host syndromes prepared before timing (GPU sampler + syndrome, copied out)
    ex = torch.empty((S, W), dtype=torch.int32, device=dev)
    ez = torch.empty((S, W), dtype=torch.int32, device=dev)
    syn_d = torch.empty((S, m), dtype=torch.uint8, device=dev)
    host_s = {}
    for ip, p in enumerate(P_LIST):
        mbbp.mbbp_sample_errors(n, S, (world * 1000 + rank * len(P_LIST) + ip) * S, SEED + 7, p,
                                mbbp.NOISE_DEPOLARIZING, ex, ez)
        for key, B, e in (("Z", BZ, ex), ("X", BX, ez)):
            mbbp.mbbp_syndrome(B, e, syn_d)
            h = torch.empty((S, m), dtype=torch.uint8, pin_memory=True)
            h.copy_(syn_d)
            host_s[(p, key)] = h
    torch.cuda.synchronize()
    out_h = {k: torch.empty((S, n), dtype=torch.uint8, pin_memory=True) for k in ("Z", "X")}
    conv_h = {k: torch.empty((S, BZ.R), dtype=torch.uint8, pin_memory=True) for k in ("Z", "X")}
    succ_h = {k: torch.empty((S,), dtype=torch.uint8, pin_memory=True) for k in ("Z", "X")}
    ws = torch.empty(mbbp.mbbp_decode_workspace_size(BZ, S), dtype=torch.uint8, device=dev)
    # double buffers: the syndromes of the next call are copied in, and the
    # results of the previous call copied out, on two copy streams while the
    # current call decodes
    syn_b = [torch.empty((S, m), dtype=torch.uint8, device=dev) for _ in range(2)]
    e_b = [torch.empty((S, n), dtype=torch.uint8, device=dev) for _ in range(2)]
    conv_b = [torch.empty((S, BZ.R), dtype=torch.uint8, device=dev) for _ in range(2)]
    succ_b = [torch.empty((S,), dtype=torch.uint8, device=dev) for _ in range(2)]
    h2d, d2h = torch.cuda.Stream(device=dev), torch.cuda.Stream(device=dev)
    ev = {k: [torch.cuda.Event(), torch.cuda.Event()] for k in ("h2d", "dec", "d2h")}
    calls = [(p, key, B) for p in P_LIST for key, B in (("Z", BZ), ("X", BX))]

    def step():
        for i, (p, key, B) in enumerate(calls):
            j = i & 1
            h2d.wait_event(ev["dec"][j])  # syndrome buffer j: its last decode is done
            with torch.cuda.stream(h2d):
                syn_b[j].copy_(host_s[(p, key)], non_blocking=True)
            ev["h2d"][j].record(h2d)
            stream.wait_event(ev["h2d"][j])
            stream.wait_event(ev["d2h"][j])  # output buffers j: their last copy-out is done
            mbbp.mbbp_decode(B, syn_b[j], llrs[p], ITERS, ALPHA, mbbp.RULE_NMS, e_b[j], conv_b[j], succ_b[j], ws,
                             stream=stream)
            ev["dec"][j].record(stream)
            d2h.wait_event(ev["dec"][j])
            with torch.cuda.stream(d2h):
                out_h[key].copy_(e_b[j], non_blocking=True)
                conv_h[key].copy_(conv_b[j], non_blocking=True)
                succ_h[key].copy_(succ_b[j], non_blocking=True)
            ev["d2h"][j].record(d2h)

    for _ in range(max(1, args.warmup)):
        step()
    torch.cuda.synchronize()
    if world > 1:
        import torch.distributed as dist
        dist.barrier()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        step()
    torch.cuda.synchronize()
    dt = time.perf_counter() - t0
    # the pipelined copies delivered the last call's results: decode it again
    # without overlap and compare
    p, key, B = calls[-1]
    ref = mbbp.decode(B, host_s[(p, key)].to(dev), llrs[p], ITERS, ALPHA)
    if not (torch.equal(ref["e_hat"].cpu(), out_h[key]) and torch.equal(ref["success"].cpu(), succ_h[key])):
        raise RuntimeError("e2e: pipelined outputs differ from a plain decode")
    if world > 1:
        import torch.distributed as dist

        from paper_2605_14170_gb300 import shard
        dt = shard.max_over_ranks(dist, dt, dev)
    shots = args.steps * len(P_LIST) * S * world
    return {"value": shots / dt, "unit": "shots/s",
            "h2d_bytes_per_step": len(P_LIST) * 2 * S * m,
            "d2h_bytes_per_step": len(P_LIST) * 2 * S * (n + BZ.R + 1)}


if __name__ == "__main__":
    main()
