#!/usr/bin/env python
"""Benchmark of the repair search.

Headline workload: the large search (4 variables, typed quasi-affine grammar, expression size <= 9,
322 884 631 700 candidates, 2^20 explicit domain points with a caller-supplied spec table).  A step is
one complete search (every size, counts and least solution) of the seed-0 instance.  The same JSON line
carries, under ``per_config``, the same measurements for the thread-binding search (config 2), the
three-hole convolution sketch (config 3, holes summed) and the batch of 4096 small instances (config 5).

``--impl reference`` times the CPU oracle on a bounded sample of the headline workload instead.
``--gpus N`` (under torchrun) runs one search per rank; ``--shard`` cuts ONE search into rank windows,
one per rank, and merges the results over the process group.
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

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "candidate_point_evals_per_s"
UNIT = "GInt-evals/s"
WORKLOADS = {
    "config2": "config2_thread_binding_matmul256_size7",
    "config3": "config3_conv2d_im2col_three_holes_size6",
    "config4": "config4_large_quasi_affine_size9_table_2p20_points",
    "config5": "config5_batch_4096_instances_size6",
}
HEADLINE = "config4"
DIVISION_COST = None

# Counters of the search kernels per step and workload, from the ncu captures in profiles/search_kernels.md (dram = dram__bytes_read.sum +
# dram__bytes_write.sum, thread_inst = smsp__thread_inst_executed.sum).  They describe the kernel sources whose hash is
# given; bench.py reports them (roofline.traffic, roofline.frac_executed) only while the sources still have that hash.
NCU_CAPTURE = {"kernel_hash": "9bc316f57788a847", "date": "2026-12-03",
               "config2": {"thread_inst": 2.369e9, "dram_bytes": 4.03e6},
               "config3": {"thread_inst": 1.714e9, "dram_bytes": 2.84e7},
               "config4": {"thread_inst": 3.404e10, "dram_bytes": 6.10e7}}


def kernel_hash() -> str:
    h = hashlib.sha256()
    csrc = os.path.join(ROOT, "paper_2505_02146_b200", "csrc")
    for name in ("xp_dev.h", "xp_device.cuh", "xp_kernels.cu", "xp_classes.cuh", "xp_join.cuh", "xp_pairs.cuh", "xp_members.cuh"):
        h.update(open(os.path.join(csrc, name), "rb").read())
    return h.hexdigest()[:16]


# ------------------------------------------------------------------------------------------
# the CPU oracle on a bounded sample of a workload (reported baseline; single thread)
# ------------------------------------------------------------------------------------------

def oracle_sample(name: str, scale: float = 1.0):
    """Times the oracle, as it stands, on a fixed part of workload ``name``; returns
    (candidate-point evaluations, seconds, description)."""
    import oracle
    from xp_instances import config2, config3, config4, config5_instance
    oracle.build()
    if name == "config5":
        n = max(1, int(48 * scale))
        t0 = time.perf_counter()
        ev = sum(oracle.repair_hole(config5_instance(0, i)).evals for i in range(n))
        return ev, time.perf_counter() - t0, f"instances 0..{n - 1} of seed 0 in full, single thread"
    sk = {"config2": config2, "config3": config3, "config4": config4}[name](0)
    K = sk.holes[0].max_size - (1 - sk.holes[0].max_size % 2)       # the largest non-empty size
    total = oracle.counts(sk.grammar, sk.holes[0].start_nt, K)[K]
    n_ranks = int({"config2": 3.0e8, "config3": 1.0e8, "config4": 2.5e8}[name] * scale)
    n_ranks = max(1, min(n_ranks, total))
    lo = min(total // 3, total - n_ranks)                            # a window away from the first block
    rr = {s: (0, 0) for s in range(1, sk.holes[0].max_size + 1)}
    rr[K] = (lo, lo + n_ranks)
    first = list(range(min(64, sk.n_points))) if sk.coords is not None else None
    t0 = time.perf_counter()
    r = oracle.repair_hole(sk, 0, rank_ranges=rr, first_points=first)
    return r.evals, time.perf_counter() - t0, f"hole 0, size-{K} ranks [{lo}, {lo + n_ranks}) of seed 0, single thread"


def cpu_baseline(name: str, scale: float = 1.0):
    ev, dt, sample = oracle_sample(name, scale)
    return {"value": ev / dt / 1e9, "unit": UNIT, "cores": 1, "kind": "oracle", "sample": sample,
            "seconds": dt, "host_cores_present": os.cpu_count()}


class ClockSampler:
    """Samples SM clocks and throttle reasons with nvidia-smi while the timed region runs."""

    def __init__(self, index: int):
        self.rows, self.proc, self.index = [], None, index

    def start(self):
        q = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
             "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
             "clocks_event_reasons.sw_power_cap")
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={q}", "--format=csv,noheader,nounits",
                                          "-i", str(self.index), "-lms", "100"], stdout=subprocess.PIPE, text=True)
            threading.Thread(target=self._read, daemon=True).start()
        except OSError:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.rows.append([x.strip() for x in line.split(",")])

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        sm = sorted(int(r[0]) for r in self.rows if r and r[0].isdigit())
        mx = [int(r[1]) for r in self.rows if len(r) > 1 and r[1].isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = [n for i, n in enumerate(names) if any(len(r) > 3 + i and r[3 + i] == "Active" for r in self.rows)]
        return {"sm_mhz": sm[len(sm) // 2] if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(sm)}


def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    name = args.workload or HEADLINE
    scale = min(1.0, 3.0 / max(1, args.steps + args.warmup))      # the whole run stays within a minute or two
    for _ in range(args.warmup):
        oracle_sample(name, scale / 8)
    evals, secs, sample = 0, 0.0, ""
    for _ in range(args.steps):
        e, dt, sample = oracle_sample(name, scale)
        evals += e
        secs += dt
    value = evals / secs / 1e9
    print(json.dumps({
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": 1e3 * secs / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "int64", "data": "synthetic",
        "config": {"workload": WORKLOADS[name], "note": "CPU oracle on a bounded rank window per step"},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": 1, "kind": "oracle", "sample": sample + " per step"},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }))


# ------------------------------------------------------------------------------------------
# one workload on the GPU
# ------------------------------------------------------------------------------------------

class Workload:
    """One config loaded on the device: ``step()`` is one complete search with everything resident;
    ``e2e_step()`` encodes grammar and sketch from host descriptors, copies the host tables, searches
    and reads the result back."""

    def __init__(self, xp, torch, name, stream, instances=4096, window=0):
        from xp_instances import config2, config3, config4, config5
        self.xp, self.torch, self.name, self.stream = xp, torch, name, stream
        self.batch = name == "config5"
        self.rr = None
        if self.batch:
            self.sks = config5(0, instances)
            self.keys = [tuple(v.hi for v in sk.grammar.variables) for sk in self.sks]
            self.grs = {}
            for sk, key in zip(self.sks, self.keys):
                if key not in self.grs:
                    self.grs[key] = xp.xp_grammar_create(sk.grammar)
            self.gdescs = {k: xp.marshal_grammar(g.model) for k, g in self.grs.items()}
            self.marshalled = xp.marshal_sketches(self.sks)      # the C descriptors, in host memory, built once
            self.loaded = xp.xp_sketch_load_batch([self.grs[k] for k in self.keys], self.sks, self.marshalled)
            self.n_points = self.sks[0].n_points
        else:
            self.sk = {"config2": config2, "config3": config3, "config4": config4}[name](0)
            self.gr = xp.xp_grammar_create(self.sk.grammar)
            self.loaded = [xp.xp_sketch_load(self.gr, self.sk)]
            self.n_points = self.sk.n_points
            if window:
                K = self.sk.holes[0].max_size - (1 - self.sk.holes[0].max_size % 2)
                self.rr = [(-1, K, 0, window)]
        self.ws = torch.empty(xp.xp_workspace_bytes(self.loaded, rank_ranges=self.rr), dtype=torch.uint8, device="cuda")

    def step(self):
        """Returns the flat list of hole results (batch: a packed array and the first hole's view)."""
        xp = self.xp
        if self.batch:
            return xp.xp_repair_batch(self.loaded, packed=True, workspace=self.ws, stream=self.stream.cuda_stream)
        return xp.xp_repair(self.loaded[0], workspace=self.ws, stream=self.stream.cuda_stream, rank_ranges=self.rr)

    @staticmethod
    def tally(res, batch):
        """(evals, candidates, kernel_ms, launches, view of the first hole) of one step's results."""
        if batch:
            import paper_2505_02146_b200 as xp
            packed, view = res
            a = xp.summaries_as_numpy(packed)
            return int(a["evals_executed"].sum()), int(a["cand_count"].sum()), view.kernel_ms, view.n_launches, view
        ev = sum(r.evals_executed for r in res)
        cand = sum(sum(r.cand_count) for r in res)
        return ev, cand, res[0].kernel_ms, res[0].n_launches, res[0]

    def e2e_step(self):
        """Host descriptors and host tables in, results out; returns (evals, h2d bytes, d2h bytes, load s, search s).
        The timed part is the library calls: grammar create, sketch load (host tables are copied to the device
        here), search, result read-back."""
        xp = self.xp
        t0 = time.perf_counter()
        if self.batch:
            grs = {k: xp.xp_grammar_create(d) for k, d in self.gdescs.items()}
            loaded = xp.xp_sketch_load_batch([grs[k] for k in self.keys], self.sks, self.marshalled)
            t1 = time.perf_counter()
            res = xp.xp_repair_batch(loaded, packed=True)
        else:
            gr = xp.xp_grammar_create(self.sk.grammar)
            loaded = [xp.xp_sketch_load(gr, self.sk)]
            t1 = time.perf_counter()
            res = xp.xp_repair(loaded[0], rank_ranges=self.rr)
        t2 = time.perf_counter()
        ev, _, _, _, view = self.tally(res, self.batch)
        infos = [xp.xp_sketch_info_get(l) for l in loaded]
        h2d = sum(int(i.load_h2d_bytes) for i in infos) + view.h2d_bytes
        d2h = sum(int(i.load_d2h_bytes) for i in infos) + view.d2h_bytes
        del loaded
        return ev, h2d, d2h, t1 - t0, t2 - t1


def measure(xp, torch, name, args, stream, flush, peak_add, barrier, sampler=None, with_cpu=True, with_e2e=True):
    """Times ``args.steps`` device-resident steps and as many end-to-end steps of one workload."""
    w = Workload(xp, torch, name, stream, instances=args.instances, window=args.window)
    for _ in range(max(3, args.warmup)):
        res = w.step()
    torch.cuda.synchronize()
    if sampler is not None:
        sampler.start()
    barrier()
    dev_ms = kern_ms = 0.0
    evals = launches = 0
    for _ in range(args.steps):
        flush.fill_(1)                                    # L2 flush (256 MiB write), outside the events
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        res = w.step()
        e1.record(stream)
        e1.synchronize()
        dev_ms += e0.elapsed_time(e1)
        ev, cand, k_ms, n_l, view = w.tally(res, w.batch)
        evals += ev
        kern_ms += k_ms
        launches += n_l
    barrier()
    clocks = sampler.stop() if sampler is not None else None
    out = {"workload": WORKLOADS[name], "dev_ms": dev_ms, "kern_ms": kern_ms, "evals": evals, "launches": launches,
           "cand": cand, "n_points": w.n_points, "view": view, "clocks": clocks, "res": res, "batch": w.batch}
    if with_e2e:
        for _ in range(2):                                # untimed: the first loads after other work are erratic
            w.e2e_step()
        torch.cuda.synchronize()
        barrier()
        e_ev = h2d = d2h = 0
        load_s = search_s = 0.0
        for _ in range(args.steps):
            flush.fill_(1)
            torch.cuda.synchronize()
            ev, a, b, ls, ss = w.e2e_step()                # (both parts end with the device idle: every call waits for it)
            e_ev += ev; h2d += a; d2h += b; load_s += ls; search_s += ss
        out["e2e_s"] = load_s + search_s
        out["e2e_evals"] = e_ev
        out["e2e"] = {"h2d": h2d // args.steps, "d2h": d2h // args.steps, "load_ms": 1e3 * load_s / args.steps,
                      "search_ms": 1e3 * search_s / args.steps}
    if with_cpu:
        out["cpu_baseline"] = cpu_baseline(name, 0.5 if name != HEADLINE else 1.0)
    return out


def roofline(m, steps, world, peak_add, peak_mad, name):
    """Both accountings of the integer-ALU roofline for one workload's measurement."""
    kern_s = m["kern_ms"] * 1e-3
    floor_ops = 2.0 * m["evals"] / world                   # one operation + one comparison per evaluation that ran
    achieved = floor_ops / kern_s / 1e9
    peak = peak_add / 1e9
    cap = NCU_CAPTURE.get(name) or {}
    fresh = NCU_CAPTURE.get("kernel_hash") == kernel_hash()
    thread_inst = cap.get("thread_inst") if fresh else None
    out = {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "G int32-op/s", "frac": achieved / peak,
           "frac_executed": (thread_inst * steps / kern_s / peak_add) if thread_inst else None,
           "frac_cost_model": (m["model_ops"] / world) / kern_s / peak_add if m.get("model_ops") else None,
           "traffic": cap.get("dram_bytes") if fresh else None,
           "division_cost": DIVISION_COST,
           "kernel": "join_kernel",
           "peak_source": "measured live: independent 32-bit add chains (xp_int32_peak); multiply-add chains reach %.0f" % (peak_mad / 1e9),
           "model": "frac: 2 x candidate-point evaluations that ran (one 32-bit operation + one comparison each) / kernel time / peak; "
                    "frac_executed: thread instructions of the search kernels per step (ncu capture %s, kernel sources %s) / live kernel time / peak; "
                    "frac_cost_model: the library's nominal_ops (a straightforward 32-bit evaluator with a 7-operation reciprocal division)"
                    % (NCU_CAPTURE.get("date"), NCU_CAPTURE.get("kernel_hash"))}
    return out


def summarise(m, steps, world, peak_add, peak_mad, name):
    value = m["evals"] / (m["dev_ms"] * 1e-3) / 1e9
    view = m["view"]
    rec = {"workload": m["workload"], "value": value, "unit": UNIT, "ms_per_step": m["dev_ms"] / steps,
           "kernel_ms_per_step": m["kern_ms"] / steps, "time_to_solution_ms": view.total_ms,
           "candidates_per_step": m["cand"], "domain_points": m["n_points"],
           "nominal_evals_per_step": m["cand"] * m["n_points"],
           "evals_executed_per_step": m["evals"] // steps,
           "candidates_per_s": m["cand"] * steps * world / (m["dev_ms"] * 1e-3),
           "gpu_launches_per_step": m["launches"] // steps,
           "roofline": roofline(m, steps, world, peak_add, peak_mad, name)}
    if "e2e" in m:
        rec["e2e"] = {"value": m["e2e_evals"] / m["e2e_s"] / 1e9, "unit": UNIT, "ms_per_step": 1e3 * m["e2e_s"] / steps,
                      "h2d_bytes_per_step": m["e2e"]["h2d"], "d2h_bytes_per_step": m["e2e"]["d2h"],
                      "load_ms": m["e2e"]["load_ms"], "search_ms": m["e2e"]["search_ms"], "l2": "flushed between steps"}
    if "cpu_baseline" in m:
        rec["cpu_baseline"] = m["cpu_baseline"]
    return rec


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-per-config", action="store_true", help="time the headline workload only")
    ap.add_argument("--shard", action="store_true",
                    help="with --gpus N: cut ONE headline search into N rank windows (one per rank) and merge the results")
    ap.add_argument("--workload", default=None, choices=sorted(WORKLOADS),
                    help="profiling aid: time this config alone (the default line's headline is config4)")
    ap.add_argument("--instances", type=int, default=4096,
                    help="profiling aid: number of instances of the config5 batch (a small case of the same kernels)")
    ap.add_argument("--window", type=int, default=0,
                    help="profiling aid: search only the first WINDOW ranks of the largest size (a small case of the same kernel)")
    args = ap.parse_args()
    if args.impl == "reference":
        run_reference(args)
        return

    import torch
    import paper_2505_02146_b200 as xp

    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    assert torch.cuda.is_available(), "bench.py needs a CUDA device: there is no CPU fallback"
    torch.cuda.set_device(local)
    dist = None
    if world > 1 or "TORCHELASTIC_RUN_ID" in os.environ:      # launched by torchrun: one rank per GPU over NCCL
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    xp.load()
    stream = torch.cuda.current_stream()
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")      # > L2 (126 MB), written between steps

    def barrier():
        if dist is not None:
            dist.barrier()
        torch.cuda.synchronize()

    peak_add, peak_mad = xp.xp_int32_peak()
    div_general, div_reciprocal = xp.xp_int_div_rate()
    global DIVISION_COST
    DIVISION_COST = {"int64_general_form": peak_add / div_general, "int32_by_constant_reciprocal_form": peak_add / div_reciprocal,
                     "unit": "32-bit add-peak operations per division, measured live (xp_int_div_rate)"}
    head = args.workload or HEADLINE
    if args.shard:
        run_shard(args, xp, torch, dist, rank, world, stream, flush, barrier)
        return

    # Independent problems shard with no data-path exchange: every rank searches its own copy of the seed-0
    # instance, so the work per GPU is the same at every N (instances of other seeds differ in cost).
    sampler = ClockSampler(local) if rank == 0 else None
    solo = world == 1
    m = measure(xp, torch, head, args, stream, flush, peak_add, barrier, sampler,
                with_cpu=solo and not args.no_cpu_baseline, with_e2e=True)
    tot = torch.tensor([m["dev_ms"], float(m["evals"]), m["e2e_s"], float(m["e2e_evals"]), m["kern_ms"]], dtype=torch.float64, device="cuda")
    if dist is not None:
        mx = tot.clone(); dist.all_reduce(mx, op=dist.ReduceOp.MAX)
        sm = tot.clone(); dist.all_reduce(sm, op=dist.ReduceOp.SUM)
        m["dev_ms"], m["e2e_s"], m["kern_ms"] = float(mx[0]), float(mx[2]), float(mx[4])
        m["evals"], m["e2e_evals"] = float(sm[1]), float(sm[3])
    if rank != 0:
        if dist is not None:
            dist.destroy_process_group()
        return
    m["model_ops"] = sum(r.nominal_ops for r in m["res"]) * args.steps * world if not m["batch"] else None
    rec = summarise(m, args.steps, world, peak_add, peak_mad, head)
    view = m["view"]
    out = {
        "metric": METRIC, "value": rec["value"], "unit": UNIT, "n_gpus": world, "steps": args.steps, "warmup": max(3, args.warmup),
        "ms_per_step": rec["ms_per_step"], "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "int64", "data": "synthetic",
        "config": {"workload": rec["workload"] + (f"_first_{args.window}_ranks_of_largest_size" if args.window else ""),
                   "candidates_per_step": rec["candidates_per_step"], "domain_points": rec["domain_points"],
                   "nominal_evals_per_step": rec["nominal_evals_per_step"],
                   "evals_executed_per_step": rec["evals_executed_per_step"],
                   "l2": "flushed between steps (256 MiB write)",
                   "time_to_solution_ms": rec["time_to_solution_ms"], "kernel_ms_per_step": rec["kernel_ms_per_step"],
                   "candidates_per_s": rec["candidates_per_s"],
                   "value_counts": "candidate-point evaluations that ran (filter tests at the first probe, exact probe checks, "
                                   "whole-domain points); candidates decided without a test are left out",
                   "parallelism": "one search per GPU, no data-path collective" if world > 1 else "one GPU"},
        "clocks": m["clocks"],
        "e2e": {k: rec["e2e"][k] for k in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step", "load_ms", "search_ms", "l2")},
        "gpu_launches": m["launches"],
        "roofline": rec["roofline"],
    }
    if not m["batch"]:
        out["config"].update({"filter_tests": view.filter_tests, "candidates_skipped": view.candidates_skipped,
                              "filter_survivors": view.filter_survivors, "probe_survivors": view.probe_survivors,
                              "least": view.least_text, "match_count": view.match_count})
    if "cpu_baseline" in rec:
        out["cpu_baseline"] = rec["cpu_baseline"]
    if solo and not args.no_per_config and args.workload is None:
        out["per_config"] = {}
        for name in ("config2", "config3", "config5"):
            mm = measure(xp, torch, name, args, stream, flush, peak_add, barrier, None,
                         with_cpu=not args.no_cpu_baseline, with_e2e=True)
            mm["model_ops"] = sum(r.nominal_ops for r in mm["res"]) * args.steps if not mm["batch"] else None
            out["per_config"][name] = summarise(mm, args.steps, 1, peak_add, peak_mad, name)
    print(json.dumps(out))
    if dist is not None:
        dist.destroy_process_group()


def run_shard(args, xp, torch, dist, rank, world, stream, flush, barrier):
    """ONE headline search cut into ``world`` contiguous rank windows per size; every rank searches its
    window, the per-hole results are merged over the process group (counts add, least rank is the
    minimum), and rank 0 compares the merged result with the stored full-size expected values."""
    from paper_2505_02146_b200.sharding import merge_results, shard_rank_windows
    from xp_instances import config4
    sk = config4(0)
    gr = xp.xp_grammar_create(sk.grammar)
    ls = xp.xp_sketch_load(gr, sk)
    counts = xp.xp_grammar_count(gr, sk.holes[0].start_nt, sk.holes[0].max_size)
    rr = shard_rank_windows(counts, world, rank, hole=0)
    ws = torch.empty(xp.xp_workspace_bytes([ls], rank_ranges=rr), dtype=torch.uint8, device="cuda")
    for _ in range(max(3, args.warmup)):
        res = xp.xp_repair(ls, workspace=ws, stream=stream.cuda_stream, rank_ranges=rr)[0]
    barrier()
    dev_ms, evals = 0.0, 0
    for _ in range(args.steps):
        flush.fill_(1)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        res = xp.xp_repair(ls, workspace=ws, stream=stream.cuda_stream, rank_ranges=rr)[0]
        if dist is not None:
            merged = merge_results(res.match_count, res.solved, res.least_size, res.least_rank)
        else:
            merged = (res.match_count, res.solved, res.least_size, res.least_rank)
        e1.record(stream)
        e1.synchronize()
        dev_ms += e0.elapsed_time(e1)
        evals += res.evals_executed
    barrier()
    tot = torch.tensor([dev_ms, float(evals)], dtype=torch.float64, device="cuda")
    if dist is not None:
        mx = tot.clone(); dist.all_reduce(mx, op=dist.ReduceOp.MAX)
        sm = tot.clone(); dist.all_reduce(sm, op=dist.ReduceOp.SUM)
        dev_ms, evals = float(mx[0]), float(sm[1])
    if rank == 0:
        gold_path = os.path.join(ROOT, "tests", "golden", "config4_seed0_full.json")
        gold = json.load(open(gold_path))["holes"][0]
        ok = (list(merged[0]) == gold["match_count"] and bool(merged[1]) == gold["solved"] and
              (not gold["solved"] or (merged[2], merged[3]) == (gold["least_size"], gold["least_rank"])))
        assert ok, "the merged result of the sharded search differs from the stored expected values"
        print(json.dumps({"metric": METRIC, "value": evals / (dev_ms * 1e-3) / 1e9, "unit": UNIT, "n_gpus": world,
                          "steps": args.steps, "warmup": max(3, args.warmup), "ms_per_step": dev_ms / args.steps,
                          "higher_is_better": True, "scaling": "strong", "vs_baseline": None, "dtype": "int64",
                          "data": "synthetic",
                          "config": {"workload": WORKLOADS["config4"], "parallelism": f"one search in {world} rank windows per size, "
                                     "merged by all-reduce (sum of counts) and all-gather (least rank)",
                                     "merged_equals_expected": True}}))
    if dist is not None:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
