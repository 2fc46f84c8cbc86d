#!/usr/bin/env python
"""Benchmark: PCTree drafting rounds on one GB300 per process.

One step = one whole drafting round of the Qwen3-4B-shaped workload
(V=151936, H=2560 bf16 head, B=16 stages, k=8, N=64, one request): B Markov
projections + log-softmax/top-k + merges, the global top-N and packing, then
the greedy accept walk against a synthetic target.  Inputs are resident in HBM
when the timed region starts; W_out (778 MB) is streamed once per stage, far
larger than L2, and the base logits rotate over 16 seeded request sets.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]

Under torchrun each rank drafts its own requests (independent replicas, no
collective on the data path); rank 0 prints one JSON line.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

from workloads import (ATTN_WORKLOADS, COMPACT_WORKLOADS, WORKLOADS,  # noqa: E402
                       draw_attention, draw_compaction, draw_head,
                       draw_request)

METRIC = ("tree-draft rounds/sec & µs/round (V=151936, B=16, N=64); "
          "% of HBM roofline")
N_SETS = 16          # rotating input sets (at most)
L2_BYTES = 129 * 1024 * 1024
FALLBACK_HBM_GBS = 6800.0


def parse_args():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="4b_b16", choices=sorted(WORKLOADS))
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-batched", action="store_true",
                    help="skip the short timing of the batched serving "
                         "workloads (8B-shaped batch 16, 14B-shaped batch 32) "
                         "that the default line carries under 'batched'")
    ap.add_argument("--no-around", action="store_true",
                    help="skip the short timing of the steps around the "
                         "round (a tree-attention layer and the compaction "
                         "at the 14B-shaped batch-32 shapes) that the default "
                         "line carries under 'around_round'")
    ap.add_argument("--e2e-logits", default="host", choices=["host", "copy"],
                    help="end-to-end leg: the kernels read each step's base "
                         "logits from the pinned host buffer over the host "
                         "link (host), or the step copies them into device "
                         "memory first (copy)")
    ap.add_argument("--mode", default="parent", choices=["parent", "shared"],
                    help="child scoring: PCTree, or the Shared-Markov control")
    ap.add_argument("--sweep", action="store_true",
                    help="k/N sweep (B in {7,16}, k in {1,2,4,8}, N in "
                         "{8..128}) on the workload's shapes, batch 1: one "
                         "JSON line per point instead of the benchmark line")
    ap.add_argument("--op", default="round",
                    choices=["round", "compact", "attention"],
                    help="round: the drafting round (the benchmark line); "
                         "compact: the accepted-row KV/hidden-state compaction "
                         "after acceptance, on --compact-workload; attention: "
                         "one tree-verification attention layer, on "
                         "--attn-workload")
    ap.add_argument("--compact-workload", default="14b_b16_bs32",
                    choices=sorted(COMPACT_WORKLOADS))
    ap.add_argument("--attn-workload", default="14b_b16_bs32",
                    choices=sorted(ATTN_WORKLOADS))
    ap.add_argument("--head-layout", default="tiled", choices=["tiled", "rowmajor"],
                    help="storage of W_out: tiled (repacked once at load with "
                         "pctree_pack_head, outside the timed region) or the "
                         "row-major [V][H] matrix")
    ap.add_argument("--path", default="auto", choices=["auto", "stagewise"],
                    help="kernel path: fused round where it applies, or the "
                         "per-stage kernels for every round")
    return ap.parse_args()


def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            return json.load(f), "measured"
    return {"hbm_gbs": FALLBACK_HBM_GBS}, "fallback"


KERNEL_SOURCES = ("paper_2608_02123_gb300/csrc/sm103_ptx.cuh",
                  "paper_2608_02123_gb300/csrc/pctree_common.cuh")


def recorded_traffic(wl, fused):
    """DRAM bytes per launch from the committed ncu summary of this kernel
    and workload, or None when the kernel changed since the capture."""
    import hashlib
    name = "round_fused" if fused else "markov_rows"
    h = hashlib.sha256()
    for f in (f"paper_2608_02123_gb300/csrc/{name}.cu", *KERNEL_SOURCES):
        with open(os.path.join(ROOT, f), "rb") as fh:
            h.update(fh.read())
    path = os.path.join(ROOT, "profiles",
                        f"{name}_kernel_qwen3_4b_V{wl.V}_H{wl.H}_B{wl.B}"
                        f"_k{wl.k}_N{wl.N}.md")
    if not os.path.exists(path):
        return None
    fields = {}
    with open(path) as fh:
        for line in fh:
            if ":" in line and line.strip().split(":")[0] in (
                    "traffic_bytes_per_launch", "kernel_sources_sha256_16"):
                key, val = line.strip().split(":", 1)
                fields[key] = val.strip()
    if fields.get("kernel_sources_sha256_16") != h.hexdigest()[:16]:
        return None
    return int(fields["traffic_bytes_per_launch"])


def stage_bytes(wl, d):
    """Algorithmic HBM bytes of stage d's Markov projection: W_out once, the
    base logits of every request at depth d, the gathered parent rows."""
    rows = wl.batch * (1 if d == 0 else wl.k)
    return wl.V * wl.H * 2 + wl.batch * wl.V * 4 + rows * wl.H * 2


def round_bytes(wl):
    return sum(stage_bytes(wl, d) for d in range(wl.B))


# ---------------------------------------------------------------------------
# clocks during the timed region
# ---------------------------------------------------------------------------

class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,"
              "clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
              "clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,"
              "clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_id):
        self.proc = None
        self.path = None
        self.gpu_id = gpu_id

    def start(self):
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            self.out = open(self.path, "w")
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "200",
                 "-i", str(self.gpu_id)], stdout=self.out,
                stderr=subprocess.DEVNULL)
        except (OSError, ValueError):
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.out.close()
        rows = []
        with open(self.path) as f:
            for line in f:
                parts = [p.strip() for p in line.split(",")]
                if len(parts) >= 9:
                    rows.append(parts)
        os.unlink(self.path)
        if not rows:
            return None
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown",
                 "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4)
                          if r[5 + i].lower() == "active"})
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(mx) if mx else None, "reasons": reasons,
                "samples": len(rows)}


# ---------------------------------------------------------------------------
# the oracle on the host cores (CPU baseline and reference arm)
# ---------------------------------------------------------------------------

def oracle_threads():
    try:
        from threadpoolctl import threadpool_info
        n = [i.get("num_threads", 0) for i in threadpool_info()
             if i.get("user_api") == "blas"]
        if n:
            return int(max(n))
    except Exception:
        pass
    return os.cpu_count() or 1


def host_cpu():
    """The host's logical CPU count and model (lscpu), for the baseline's
    record."""
    model = None
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True,
                             timeout=10).stdout
        for line in out.splitlines():
            if line.strip().startswith("Model name:"):
                model = line.split(":", 1)[1].strip()
                break
    except (OSError, subprocess.SubprocessError):
        pass
    return {"nproc": os.cpu_count(), "model": model}


class OracleRunner:
    """Runs the oracle's drafting round on the workload's rounds (whole
    rounds, or the first `stages` of the B stages of each)."""

    def __init__(self, wl, E_in, W_out_bits, sets):
        from oracle import pctree_oracle as O
        self.O, self.wl, self.E_in, self.sets = O, wl, E_in, sets
        self.W = O.as_f64(W_out_bits, wl.weight_dtype)   # weights load once

    def run(self, i, stages=None, hint=None):
        L, root = self.sets[i % len(self.sets)]
        s = self.wl.B if stages is None else stages
        return self.O.draft(L[:s], self.E_in, self.W, root, s, self.wl.k,
                            self.wl.N, mode=self.wl.mode, hint=hint)


def markov_rows(wl, stages):
    """Markov rows the first `stages` stages of a round evaluate: one per
    request at stage 0, then one per frontier parent (k per request), or one
    chain row per request in the Shared-Markov control.  The oracle's cost
    is proportional to these rows (each is a vocabulary-wide projection and
    selection), so partial-round samples are scaled to whole rounds by them."""
    per_stage = 1 if wl.mode == "shared" else wl.k
    return wl.batch * (1 + (stages - 1) * per_stage) if stages > 0 else 0


def tree_hint(O, host, r=0):
    """The GPU round's decisions (children, frontiers, kept set) rebuilt from
    its candidate pool, for the oracle's near-tie replay."""
    n = int(host["n_nodes"][r])
    tok, par = host["tokens"][r], host["parent"][r]
    paths = []
    for a in range(n):
        paths.append(() if a == 0 else paths[par[a]] + (int(tok[a]),))
    return O.choices_from_pool(host["pool_token"][r], host["pool_parent"][r],
                               host["pool_token"].shape[1], set(paths))


def cpu_baseline(runner, wl, gpu_trees, budget_s=12.0):
    """The oracle, as it stands, on whole rounds of the benchmark's input sets
    (request 0 of each), for about `budget_s` seconds on the host cores.
    Each round replays the GPU round's near-tie decisions (``hint``; the
    replay only engages where the two differ), so the same runs also check
    the benchmark's own trees against the oracle."""
    O = runner.O
    times, ambiguous, max_err, equal = [], 0, 0.0, True
    t_start = time.perf_counter()
    i = 0
    while i < len(gpu_trees) and (i < 2 or time.perf_counter() - t_start < budget_s):
        host = gpu_trees[i]
        t0 = time.perf_counter()
        rnd = runner.run(i, hint=tree_hint(O, host))
        times.append(time.perf_counter() - t0)
        t = rnd.tree
        ambiguous += rnd.n_ambiguous
        n = t.n_nodes
        equal &= (int(host["n_nodes"][0]) == n and
                  all((host[f][0] == getattr(t, f)).all()
                      for f in ("tokens", "parent", "depth", "mask",
                                "retrieve")))
        fin = np.isfinite(t.logp[:n])
        if fin.any():
            max_err = max(max_err, float(np.abs(host["logp"][0][:n][fin]
                                                - t.logp[:n][fin]).max()))
        i += 1
    dt = sum(times)
    return {"value": len(times) / dt, "unit": "rounds/s",
            "cores": oracle_threads(), "host": host_cpu(), "kind": "oracle",
            "sample": f"{len(times)} whole oracle rounds of {wl.name} "
                      f"(input sets 0..{len(times) - 1}, request 0), "
                      f"{dt:.1f} s, {dt / len(times):.2f} s per round",
            "oracle_check": {"rounds": len(times), "trees_equal": bool(equal),
                             "ambiguous": ambiguous,
                             "max_abs_logp_err": max_err}}


def run_reference(args, wl, rank, world, budget_s=180.0):
    """The oracle on the host cores, one drafting round per step.  Steps are
    whole rounds when K + W of them fit in ``budget_s``; otherwise each step
    runs the first stages of a round, scaled to whole rounds by Markov rows."""
    if rank != 0:
        return
    E_in, W_out = draw_head(wl)
    sets = []
    for r in range(4):
        L, root, _, _ = draw_request(wl.with_(batch=N_SETS), r)
        sets.append((L, root))
    runner = OracleRunner(wl, E_in, W_out, sets)
    t0 = time.perf_counter()
    runner.run(0)                                    # first warm-up: a whole round
    t_round = time.perf_counter() - t0
    stages = wl.B
    while stages > 1 and (args.steps + args.warmup) * t_round * \
            markov_rows(wl, stages) / markov_rows(wl, wl.B) > budget_s:
        stages -= 1
    scale = markov_rows(wl, wl.B) / markov_rows(wl, stages)
    for i in range(1, args.warmup):
        runner.run(i, stages)
    t0 = time.perf_counter()
    for i in range(args.steps):
        runner.run(i, stages)
    dt = time.perf_counter() - t0
    value = args.steps / scale / dt
    step = ("one whole oracle round (all {} stages)".format(wl.B)
            if stages == wl.B else
            f"the oracle's first {stages} of {wl.B} stages of a round, "
            f"scaled to whole rounds by Markov rows "
            f"({markov_rows(wl, wl.B)}/{markov_rows(wl, stages)}); a whole "
            f"round took {t_round:.2f} s")
    line = {
        "metric": METRIC, "value": value, "unit": "rounds/s",
        "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": dt * 1e3 / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic", "impl": "reference",
        "config": {"workload": wl.name, "V": wl.V, "H": wl.H, "B": wl.B,
                   "k": wl.k, "N": wl.N, "batch": wl.batch, "step": step},
        "cpu_baseline": {"value": value, "unit": "rounds/s",
                         "cores": oracle_threads(), "host": host_cpu(),
                         "kind": "oracle",
                         "sample": f"{args.steps} steps, each {step}"},
        "e2e": {"value": value, "unit": "rounds/s", "h2d_bytes_per_step": 0,
                "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


# ---------------------------------------------------------------------------
# the CUDA path
# ---------------------------------------------------------------------------

# ---------------------------------------------------------------------------
# multi-rank plumbing: independent replicas, no collective on the data path
# ---------------------------------------------------------------------------

def rank_requests(rank, world, n_sets, batch):
    """Request indices of every input set on this rank.  Ranks draw disjoint
    requests (each GPU drafts its own), so the job's requests are
    ``world * n_sets * batch`` distinct ones."""
    per_rank = n_sets * batch
    return [[rank * per_rank + i * batch + b for b in range(batch)]
            for i in range(n_sets)]


def max_over_ranks(values, world, device=None):
    """Element-wise maximum of per-rank timings (the slowest rank sets the
    job's time)."""
    if world == 1:
        return [float(v) for v in values]
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(v) for v in values], dtype=torch.float64,
                     device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return [float(v) for v in t.tolist()]


def job_rounds_per_s(ms_max, steps, world, batch):
    """Whole-job throughput: every rank's rounds over the slowest rank's
    time."""
    return steps * world * batch / (ms_max / 1e3)


def slow_steps(step_ms, most=16):
    """[index, ms] of the steps that took over 1.3 times the median."""
    limit = 1.3 * statistics.median(step_ms)
    return [[i, x] for i, x in enumerate(step_ms) if x > limit][:most]


def run_ours(args, wl, rank, world, local_rank):
    import torch
    import torch.distributed as dist

    from paper_2608_02123_gb300 import pctree as P

    dev = torch.device("cuda", local_rank)
    torch.cuda.set_device(dev)
    E_host, W_host = draw_head(wl)
    if wl.weight_dtype == "bf16":
        E = torch.from_numpy(E_host.view(np.int16)).to(dev).view(torch.bfloat16)
        W = torch.from_numpy(W_host.view(np.int16)).to(dev).view(torch.bfloat16)
    else:
        E = torch.from_numpy(E_host).to(dev)
        W = torch.from_numpy(W_host).to(dev)
    # rotating input sets, each a whole batch of distinct requests; enough
    # sets that their base logits exceed the L2 three times over
    batch_bytes = wl.batch * wl.B * wl.V * 4
    n_sets = max(2, min(N_SETS, -(-3 * L2_BYTES // batch_bytes)))
    many = wl.with_(batch=n_sets * wl.batch * world)
    sets = []
    for ids in rank_requests(rank, world, n_sets, wl.batch):
        reqs = [draw_request(many, q) for q in ids]
        sets.append((np.stack([q[0] for q in reqs]),
                     np.asarray([q[1] for q in reqs], np.int32),
                     np.stack([q[2] for q in reqs])))
    L_dev = [torch.from_numpy(L).to(dev) for L, _, _ in sets]
    root_dev = [torch.from_numpy(root).to(dev) for _, root, _ in sets]
    greedy_dev = [torch.from_numpy(g.astype(np.int64)).to(dev)
                  for _, _, g in sets]
    layout = args.head_layout if wl.weight_dtype == "bf16" else "rowmajor"
    cfg = P.make_config(wl.V, wl.H, wl.B, wl.k, wl.N, wl.batch, wl.pos_offset,
                        wl.weight_dtype, wl.mode, layout)
    if layout == "tiled":
        # the weights are fixed: repacked once, as a serving process does at
        # load; the row-major copy is released
        W = P.pack_head(cfg, W)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
    path = P.PATH_AUTO if args.path == "auto" else P.PATH_STAGEWISE
    P.pctree_set_path(path)
    num_sms = torch.cuda.get_device_properties(dev).multi_processor_count
    fused = P.runs_fused_round(cfg, path, num_sms)
    dr = P.Drafter(cfg, dev)
    stream = torch.cuda.current_stream()

    def target_of(i, tree=None):
        # synthetic target model: node i at depth t wants g[t] as its child
        depth = (dr.tree if tree is None else tree).depth.long().clamp_min(0)
        return torch.gather(greedy_dev[i % n_sets], 1, depth).to(torch.int32)

    def step(i):
        dr.draft(L_dev[i % n_sets], E, W, root_dev[i % n_sets], stream)
        dr.accept(target_of(i), stream)

    for i in range(args.warmup):
        step(i)
    torch.cuda.synchronize()
    dr.check_status()
    if world > 1:
        dist.barrier()

    gpu_index = os.environ.get("CUDA_VISIBLE_DEVICES", str(local_rank))
    gpu_index = gpu_index.split(",")[local_rank] if "," in gpu_index else gpu_index
    clocks = ClockSampler(gpu_index)
    clocks.start()
    time.sleep(0.3)  # first sample lands inside the timed work below
    start = torch.cuda.Event(enable_timing=True)
    end = torch.cuda.Event(enable_timing=True)
    # per-step events (draft, accept) inside the bracketed timing, for the
    # distribution of round times and the accept call on its own
    marks = [[torch.cuda.Event(enable_timing=True) for _ in range(4)]
             for _ in range(args.steps)]
    torch.cuda.synchronize()
    start.record(stream)
    for i in range(args.steps):
        m = marks[i]
        m[0].record(stream)
        dr.draft(L_dev[i % n_sets], E, W, root_dev[i % n_sets], stream)
        m[1].record(stream)
        tgt = target_of(i)
        m[2].record(stream)
        dr.accept(tgt, stream)
        m[3].record(stream)
    end.record(stream)
    torch.cuda.synchronize()
    draft_us = sorted(m[0].elapsed_time(m[1]) * 1e3 for m in marks)
    accept_us = [m[2].elapsed_time(m[3]) * 1e3 for m in marks]
    dr.check_status()
    ms = start.elapsed_time(end)
    # the projection launches on their own, in rounds outside the timed region:
    # the events around them keep a kernel from being launched while its
    # predecessor finishes
    prof_steps = min(args.steps, 20)
    P.pctree_profile_enable(True)
    for i in range(prof_steps):
        dr.draft(L_dev[i % n_sets], E, W, root_dev[i % n_sets], stream)
    torch.cuda.synchronize()
    launches, proj_ms = P.pctree_profile_collect()
    P.pctree_profile_enable(False)
    dr.check_status()

    # end to end through the public API: pinned host inputs in, tree out
    L_host = [torch.from_numpy(L).pin_memory() for L, _, _ in sets]
    root_host = [torch.from_numpy(root).pin_memory() for _, root, _ in sets]
    # the tree and the acceptance outputs share one device buffer: one copy
    # brings every result back
    out_host = torch.empty(dr.tree.blob.shape, dtype=torch.uint8, pin_memory=True)
    h2d = L_host[0].numel() * 4 + root_host[0].numel() * 4
    d2h = out_host.numel()
    L_stage = torch.empty_like(L_dev[0])
    root_stage = torch.empty_like(root_dev[0])
    def e2e_step(i, zero_copy):
        if zero_copy:
            # the kernels read the pinned host inputs as they need them
            L_in, root_in = L_host[i % n_sets], root_host[i % n_sets]
        else:
            L_stage.copy_(L_host[i % n_sets], non_blocking=True)
            root_stage.copy_(root_host[i % n_sets], non_blocking=True)
            L_in, root_in = L_stage, root_stage
        dr.draft(L_in, E, W, root_in, stream)
        dr.accept(target_of(i), stream)
        out_host.copy_(dr.tree.blob, non_blocking=True)
        stream.synchronize()   # the caller reads the tree before the next round

    def e2e_time(zero_copy):
        # every input set once before timing: the GPU's first reads of a pinned
        # buffer go through address translations it has not seen
        for i in range(max(3, n_sets)):
            e2e_step(i, zero_copy)
        # each step's host time beside the total: a few stalled steps (of the
        # host or the link) in a short run would set the mean alone
        step_ms = []
        e_start = torch.cuda.Event(enable_timing=True)
        e_end = torch.cuda.Event(enable_timing=True)
        e_start.record(stream)
        for i in range(args.steps):
            t0 = time.perf_counter()
            e2e_step(i, zero_copy)
            step_ms.append((time.perf_counter() - t0) * 1e3)
        e_end.record(stream)
        torch.cuda.synchronize()
        return e_start.elapsed_time(e_end), step_ms

    # the headline e2e as --e2e-logits says, and the other way beside it
    zero_copy = args.e2e_logits == "host"
    e2e_ms, e2e_steps = e2e_time(zero_copy)
    e2e_other_ms, _ = e2e_time(not zero_copy)
    clk = clocks.stop()

    # outside the timed regions: one round per input set with its candidate
    # pool, for the mean acceptance length on the synthetic target and for
    # the oracle's check of the benchmark's own trees
    check = P.Drafter(cfg, dev, with_pool=True)
    accepted, gpu_trees = [], []
    for i in range(n_sets):
        check.draft(L_dev[i], E, W, root_dev[i], stream)
        check.accept(target_of(i, check.tree), stream)
        torch.cuda.synchronize()
        check.check_status()
        accepted += check.accepted_len.cpu().tolist()
        gpu_trees.append(check.tree.to_host())
    mean_tau = 1.0 + float(np.mean(accepted))     # tau counts the bonus token

    ms, e2e_ms, e2e_other_ms = max_over_ranks([ms, e2e_ms, e2e_other_ms], world, dev)
    if rank != 0:
        return

    value = job_rounds_per_s(ms, args.steps, world, wl.batch)
    peaks, peak_kind = measured_peaks()
    peak = float(peaks["hbm_gbs"])
    bytes_round = round_bytes(wl)
    proj_bytes = prof_steps * bytes_round          # those launches' bytes
    achieved = proj_bytes / (proj_ms / 1e3) / 1e9 if proj_ms > 0 else None
    us_round = ms * 1e3 / args.steps
    kernels_per_step = P.kernels_per_round(cfg, path, num_sms) + 1    # + accept
    line = {
        "metric": METRIC, "value": value, "unit": "rounds/s",
        "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": ms / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "bf16",
        "data": "synthetic (seeded Qwen3-4B-shaped logits, random-init head)",
        "config": {"workload": wl.name, "V": wl.V, "H": wl.H, "B": wl.B,
                   "k": wl.k, "N": wl.N, "batch": wl.batch,
                   "parallelism": f"replicas x{world}",
                   "kernel_path": args.path, "mode": wl.mode,
                   "head_layout": (f"{layout} (W_out repacked once at load by "
                                   "pctree_pack_head, outside the timed region)"
                                   if layout == "tiled" else layout),
                   "l2": f"inputs larger than L2: W_out "
                         f"({wl.V * wl.H * (2 if wl.weight_dtype == 'bf16' else 4) / 1e6:.0f} MB) "
                         f"streamed per stage; base logits rotate over "
                         f"{n_sets} input sets"},
        "us_per_round": us_round,
        "round_hbm_fraction": (bytes_round / (us_round * 1e-6) / 1e9) / peak,
        "roofline": {"bound": "hbm",
                     "kernel": ("round_fused_kernel" if fused
                                else "markov_rows_kernel"),
                     "achieved": achieved, "peak": peak, "unit": "GB/s",
                     "frac": achieved / peak if achieved else None,
                     "peak_source": peak_kind,
                     "launches": launches,
                     "avg_launch_us": proj_ms * 1e3 / launches if launches else None,
                     "traffic": (recorded_traffic(wl, fused) if layout == "tiled" and
                                 wl.name == f"qwen3_4b_V{wl.V}_H{wl.H}_B{wl.B}_k{wl.k}_N{wl.N}_bs1"
                                 else None)},
        "draft_us": {"p10": draft_us[len(draft_us) // 10],
                     "p50": draft_us[len(draft_us) // 2],
                     "p90": draft_us[(9 * len(draft_us)) // 10]},
        "accept_us": statistics.mean(accept_us),
        "mean_tau_synthetic": mean_tau,
        "mean_tau_note": f"mean accepted length + 1 over the {n_sets} input "
                         f"sets' rounds against the synthetic target (a "
                         f"property of the input generator, not of a model)",
        "e2e": {"value": job_rounds_per_s(e2e_ms, args.steps, world, wl.batch),
                "unit": "rounds/s",
                "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h,
                "step_ms": {"p50": statistics.median(e2e_steps),
                            "max": max(e2e_steps),
                            "slow": slow_steps(e2e_steps)},
                "inputs": ("base logits and root tokens in pinned host memory, "
                           "read by the kernels over the host link as they need "
                           "them (no copy)" if zero_copy else
                           "base logits and root tokens copied to device memory "
                           "each step (cudaMemcpyAsync)"),
                "outputs": "tree and acceptance results in one device buffer, "
                           "one copy back per step",
                ("with_input_copy" if zero_copy else "without_input_copy"): {
                    "value": job_rounds_per_s(e2e_other_ms, args.steps, world, wl.batch),
                    "unit": "rounds/s",
                    "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h}},
        "gpu_launches": kernels_per_step * args.steps,
        "clocks": clk,
    }
    if world == 1 and not args.no_batched and args.workload == "4b_b16":
        line["batched"] = measure_batched(dev, gpu_index, layout)
    if world == 1 and not args.no_around and args.workload == "4b_b16":
        # the steps of a serving round around the draft, at the 14B-shaped
        # batch-32 serving shapes: one verification attention layer and the
        # compaction after acceptance
        line["around_round"] = [
            measure_attention("14b_b16_bs32", local_rank, 2000, 10, gpu_index),
            measure_compact("14b_b16_bs32", local_rank, 8000, 10, gpu_index)]
    if world == 1 and not args.no_cpu_baseline:
        runner = OracleRunner(wl, E_host, W_host,
                              [(L[0], int(root[0])) for L, root, _ in sets])
        base = cpu_baseline(runner, wl, gpu_trees)
        line["cpu_baseline"] = base
        line["ambiguous"] = base["oracle_check"]["ambiguous"]
    print(json.dumps(line), flush=True)


# ---------------------------------------------------------------------------
# batched serving rounds, timed briefly beside the headline
# ---------------------------------------------------------------------------

BATCHED = ("8b_b7_bs16", "14b_b16_bs32")


def round_flops(wl):
    """Tensor-core flops of a round's Markov projections: 2 H V per Markov
    row."""
    rows = sum(wl.batch * (1 if d == 0 else wl.k) for d in range(wl.B))
    return 2.0 * wl.H * wl.V * rows


def measure_batched(dev, gpu_index, layout, steps=10, warmup=3):
    """Each batched workload: W + K whole rounds (inputs resident, base
    logits rotating over sets that together exceed 3 x L2), CUDA events on
    the launching stream, clocks sampled meanwhile.  The roofline is HBM
    (algorithmic bytes) or tensor (projection flops) by whichever takes
    longer at the measured peaks; the sustained bf16 rate is the one for a
    round of several milliseconds."""
    import torch

    from paper_2608_02123_gb300 import pctree as P

    peaks, src = measured_peaks()
    hbm = float(peaks["hbm_gbs"])
    tc = float(peaks.get("bf16_tflops_sustained", peaks.get("bf16_tflops", 1700.0)))
    out = []
    stream = torch.cuda.current_stream()
    num_sms = torch.cuda.get_device_properties(dev).multi_processor_count
    for name in BATCHED:
        wl = WORKLOADS[name]
        E_host, W_host = draw_head(wl)
        E = torch.from_numpy(E_host.view(np.int16)).to(dev).view(torch.bfloat16)
        W = torch.from_numpy(W_host.view(np.int16)).to(dev).view(torch.bfloat16)
        del E_host, W_host
        set_bytes = wl.batch * wl.B * wl.V * 4
        n_sets = max(2, -(-3 * L2_BYTES // set_bytes))
        many = wl.with_(batch=n_sets * wl.batch)
        L_dev, root_dev = [], []
        for i in range(n_sets):
            reqs = [draw_request(many, i * wl.batch + b) for b in range(wl.batch)]
            L_dev.append(torch.from_numpy(np.stack([q[0] for q in reqs])).to(dev))
            root_dev.append(torch.tensor([q[1] for q in reqs], dtype=torch.int32,
                                         device=dev))
        cfg = P.make_config(wl.V, wl.H, wl.B, wl.k, wl.N, wl.batch, 0, "bf16",
                            "parent", layout)
        if layout == "tiled":
            W = P.pack_head(cfg, W)
        dr = P.Drafter(cfg, dev)
        for i in range(warmup):
            dr.draft(L_dev[i % n_sets], E, W, root_dev[i % n_sets], stream)
        torch.cuda.synchronize()
        dr.check_status()
        clocks = ClockSampler(gpu_index)
        clocks.start()
        time.sleep(0.3)
        start = torch.cuda.Event(enable_timing=True)
        end = torch.cuda.Event(enable_timing=True)
        start.record(stream)
        for i in range(steps):
            dr.draft(L_dev[i % n_sets], E, W, root_dev[i % n_sets], stream)
        end.record(stream)
        torch.cuda.synchronize()
        clk = clocks.stop()
        dr.check_status()
        us = start.elapsed_time(end) * 1e3 / steps
        nbytes, flops = round_bytes(wl), round_flops(wl)
        t_hbm, t_tc = nbytes / hbm / 1e3, flops / tc / 1e6   # µs
        bound = "hbm" if t_hbm >= t_tc else "tensor"
        out.append({
            "workload": wl.name, "batch": wl.batch, "steps": steps,
            "head_layout": layout,
            "warmup": warmup, "us_per_round": us,
            "rounds_per_s": 1e6 / us, "request_rounds_per_s": wl.batch * 1e6 / us,
            "bound": bound, "roofline_us": max(t_hbm, t_tc),
            "frac": max(t_hbm, t_tc) / us,
            "achieved": {"GB/s": nbytes / us / 1e3, "TFLOP/s": flops / us / 1e6},
            "peak": {"GB/s": hbm, "TFLOP/s": tc, "source": src,
                     "tensor": "sustained bf16"},
            "gpu_launches": steps * P.kernels_per_round(cfg, num_sms=num_sms),
            "clocks": clk})
        del E, W, L_dev, dr
        torch.cuda.empty_cache()
    return out


# ---------------------------------------------------------------------------
# k / N sweep (the shapes of the paper's ablations, Sec. 5.4)
# ---------------------------------------------------------------------------

SWEEP_B = (7, 16)
SWEEP_K = (1, 2, 4, 8)
SWEEP_N = (8, 16, 24, 32, 48, 64, 96, 128)


def run_sweep(args, wl, local_rank):
    import torch

    from paper_2608_02123_gb300 import pctree as P

    dev = torch.device("cuda", local_rank)
    torch.cuda.set_device(dev)
    base = wl.with_(B=max(SWEEP_B), batch=1)
    E_host, W_host = draw_head(base)
    E = torch.from_numpy(E_host.view(np.int16)).to(dev).view(torch.bfloat16)
    W = torch.from_numpy(W_host.view(np.int16)).to(dev).view(torch.bfloat16)
    layout = args.head_layout
    if layout == "tiled":
        # one tiled copy serves every (B, k, N) point (it depends on V, H only)
        W = P.pack_head(P.make_config(base.V, base.H, 1, 1, 1, 1, 0, "bf16", "parent",
                                      "tiled"), W)
        torch.cuda.synchronize()
    n_sets = N_SETS
    many = base.with_(batch=n_sets)
    reqs = [draw_request(many, i) for i in range(n_sets)]
    peak = float(measured_peaks()[0]["hbm_gbs"])
    steps = max(args.steps // 4, 10)
    stream = torch.cuda.current_stream()
    num_sms = torch.cuda.get_device_properties(dev).multi_processor_count
    for B in SWEEP_B:
        L_dev = [torch.from_numpy(np.ascontiguousarray(q[0][None, :B])).to(dev)
                 for q in reqs]
        root_dev = [torch.tensor([q[1]], dtype=torch.int32, device=dev)
                    for q in reqs]
        g_dev = [torch.from_numpy(np.concatenate([q[2][:B], q[2][-1:]])[None]
                                  .astype(np.int64)).to(dev) for q in reqs]
        for k in SWEEP_K:
            for N in SWEEP_N:
                wk = base.with_(B=B, k=k, N=N)
                cfg = P.make_config(wk.V, wk.H, B, k, N, 1, 0, "bf16", wk.mode, layout)
                dr = P.Drafter(cfg, dev)
                taus = []

                def step(i, keep=False):
                    dr.draft(L_dev[i % n_sets], E, W, root_dev[i % n_sets], stream)
                    depth = dr.tree.depth.long().clamp_min(0)
                    tgt = torch.gather(g_dev[i % n_sets], 1, depth).to(torch.int32)
                    dr.accept(tgt, stream)
                    if keep:
                        taus.append(dr.accepted_len.clone())

                for i in range(3):
                    step(i)
                torch.cuda.synchronize()
                start = torch.cuda.Event(enable_timing=True)
                end = torch.cuda.Event(enable_timing=True)
                start.record(stream)
                for i in range(steps):
                    step(i, keep=True)
                end.record(stream)
                torch.cuda.synchronize()
                dr.check_status()
                ms = start.elapsed_time(end) / steps
                tau = float(torch.stack(taus).float().mean()) + 1.0
                print(json.dumps({
                    "sweep": "kN", "workload": wk.name, "mode": wk.mode,
                    "head_layout": layout, "rounds": steps,
                    "B": B, "k": k, "N": N, "us_per_round": ms * 1e3,
                    "rounds_per_s": 1e3 / ms,
                    "round_hbm_fraction": round_bytes(wk) / (ms * 1e-3) / 1e9 / peak,
                    "fused": P.runs_fused_round(cfg, num_sms=num_sms),
                    "mean_tau_synthetic_target": tau}), flush=True)


def compact_bytes(cw, acc, lens):
    """Algorithmic bytes of one compaction: every moved cache row read and
    written once (nodes with a[j] == j at the head of the path stay), every
    gathered hidden-state row read and written once."""
    total = 0
    for r in range(cw.batch):
        L = int(lens[r])
        j = 1
        while j <= L and acc[r, j] == j:
            j += 1
        total += (L + 1 - j) * cw.layers * cw.planes * cw.row_bytes * 2
        total += (L + 1) * cw.hidden_bytes * 2
    return total


def measure_compact(name, local_rank, steps, warmup, gpu_index=None):
    """Accepted-row compaction (the step after acceptance) on one GPU: a
    cache of the workload's shape resident in HBM, accepted paths and
    prefix lengths rotating over 16 seeded sets, so a launch's rows were
    last touched 15 launches (and, at the large workloads, over 1 GB of
    other rows) earlier: inputs larger than L2, no flush.  Returns the
    measurement as a dict."""
    import torch

    from paper_2608_02123_gb300 import pctree as P

    cw = COMPACT_WORKLOADS[name]
    dev = torch.device("cuda", local_rank)
    torch.cuda.set_device(dev)
    gen = torch.Generator(device=dev)
    gen.manual_seed(cw.seed)
    cache = torch.randint(0, 256, (cw.cache_bytes(),), dtype=torch.uint8,
                          device=dev, generator=gen)
    hin = torch.randint(0, 256, (cw.batch, cw.N, cw.hidden_bytes),
                        dtype=torch.uint8, device=dev, generator=gen)
    hout = torch.zeros((cw.batch, cw.B + 1, cw.hidden_bytes), dtype=torch.uint8,
                       device=dev)
    sets = [draw_compaction(cw, seed=cw.seed * 1000 + i, fill=False)
            for i in range(N_SETS)]
    acc = [torch.from_numpy(c.accepted_idx).to(dev) for c in sets]
    lens = [torch.from_numpy(c.accepted_len).to(dev) for c in sets]
    pre = [torch.from_numpy(c.prefix_len).to(dev) for c in sets]
    nbytes = [compact_bytes(cw, c.accepted_idx, c.accepted_len) for c in sets]
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    lay = P.compact_layout(cw.batch, cw.B, cw.N, cw.layers, cw.planes,
                           cw.slots, cw.row_bytes, hidden_bytes=cw.hidden_bytes)
    stream = torch.cuda.current_stream()

    def step(i, s=None):
        j = i % N_SETS
        P.pctree_compact(lay, acc[j], lens[j], pre[j], cache, hin, hout,
                         status, s if s is not None else stream)

    for i in range(max(warmup, 3)):
        step(i)
    torch.cuda.synchronize()
    # A launch moves a few MB in a few microseconds, less than a Python
    # caller takes to issue it: the timed launches are replayed from a CUDA
    # graph (one capture of the 16 path sets) so that the host's launch
    # rate does not set the measured rate.
    graph = torch.cuda.CUDAGraph()
    cap = torch.cuda.Stream()
    cap.wait_stream(stream)
    with torch.cuda.graph(graph, stream=cap):
        for i in range(N_SETS):
            step(i, torch.cuda.current_stream())
    torch.cuda.synchronize()
    reps = max(1, steps // N_SETS)
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    start = torch.cuda.Event(enable_timing=True)
    end = torch.cuda.Event(enable_timing=True)
    clocks = ClockSampler(local_rank if gpu_index is None else gpu_index)
    clocks.start()
    start.record(stream)
    for _ in range(reps):
        graph.replay()
    end.record(stream)
    torch.cuda.synchronize()
    clk = clocks.stop()
    steps = reps * N_SETS
    if int(status.item()) != 0:
        raise RuntimeError(f"pctree_compact status {int(status.item())}")
    total_ms = start.elapsed_time(end)
    moved = sum(nbytes[i % N_SETS] for i in range(steps))
    peaks, src = measured_peaks()
    peak = float(peaks["hbm_gbs"])
    achieved = moved / (total_ms * 1e-3) / 1e9
    us = total_ms * 1e3 / steps
    del cache, hin, hout, graph
    torch.cuda.empty_cache()
    return {
        "metric": "accepted-row compaction µs/round (KV planes + hidden states)",
        "value": us, "unit": "us/round", "higher_is_better": False,
        "n_gpus": 1, "steps": steps, "warmup": max(warmup, 3),
        "dtype": "u8", "data": "synthetic (seeded cache bytes and accepted paths)",
        "config": {"workload": cw.name, "layers": cw.layers,
                   "planes": cw.planes, "row_bytes": cw.row_bytes,
                   "hidden_bytes": cw.hidden_bytes, "B": cw.B, "N": cw.N,
                   "batch": cw.batch, "slots": cw.slots,
                   "l2": "16 rotating path sets; rows larger than L2 between reuses",
                   "launch": "timed launches replayed from a CUDA graph of the 16 path sets"},
        "bytes_per_round": moved / steps,
        "roofline": {"bound": "hbm", "kernel": "compact_kernel",
                     "achieved": achieved, "peak": peak, "unit": "GB/s",
                     "frac": achieved / peak, "peak_source": src,
                     "traffic": None},
        "gpu_launches": steps, "clocks": clk}


def run_compact(args, local_rank):
    print(json.dumps(measure_compact(args.compact_workload, local_rank,
                                     args.steps, args.warmup)), flush=True)


def attention_work(ai):
    """Algorithmic bytes and flops of one tree-attention layer: K and V of
    every request's prefix and tree read once per KV head, Q read and the
    output written once; 4 * D flops per (node, query head, allowed key)
    pair (the scores and the weighted sum)."""
    aw = ai.aw
    nbytes, flops = 0, 0
    for r in range(aw.batch):
        T, n = int(ai.prefix_len[r]), int(ai.n_nodes[r])
        nbytes += (T + n) * aw.Hkv * aw.D * 2 * 2
        nbytes += n * aw.Hq * aw.D * 2 * 2
        depth = np.zeros(aw.N, dtype=np.int64)
        for i in range(1, n):
            depth[i] = depth[ai.parent[r, i]] + 1
        keys = T + depth[:n] + 1
        flops += int(keys.sum()) * aw.Hq * 4 * aw.D
    return nbytes, flops


def measure_attention(name, local_rank, steps, warmup, gpu_index=None):
    """One tree-verification attention layer (the target's forward that
    verifies the packed tree) on one GPU: the workload's caches resident in
    HBM, rotated over enough copies that a launch's K/V were last read more
    than 3 x L2 earlier.  Returns the measurement as a dict."""
    import torch

    from paper_2608_02123_gb300 import pctree as P

    aw = ATTN_WORKLOADS[name]
    dev = torch.device("cuda", local_rank)
    torch.cuda.set_device(dev)
    ai = draw_attention(aw)

    def up(bits):
        return torch.from_numpy(bits.view(np.int16)).to(dev).view(torch.bfloat16)

    q, k, v = up(ai.q), up(ai.k), up(ai.v)
    kv_bytes = 2 * k.numel() * 2
    n_sets = max(1, min(64, -(-3 * L2_BYTES // kv_bytes)))
    ks = [k] + [k.clone() for _ in range(n_sets - 1)]
    vs = [v] + [v.clone() for _ in range(n_sets - 1)]
    pre = torch.from_numpy(ai.prefix_len).to(dev)
    nn = torch.from_numpy(ai.n_nodes).to(dev)
    par = torch.from_numpy(ai.parent).to(dev)
    out = torch.empty_like(q)
    cfg = P.attn_config(aw.batch, aw.N, aw.Hq, aw.Hkv, aw.slots)
    nb = P.pctree_tree_attention_workspace_bytes(cfg)
    ws = torch.empty(max(nb, 1), dtype=torch.uint8, device=dev) if nb else None
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    stream = torch.cuda.current_stream()

    def step(i):
        P.pctree_tree_attention(cfg, q, ks[i % n_sets], vs[i % n_sets], pre, nn,
                                par, out, ws, status, stream)

    for i in range(max(warmup, 3)):
        step(i)
    torch.cuda.synchronize()
    start = torch.cuda.Event(enable_timing=True)
    end = torch.cuda.Event(enable_timing=True)
    clocks = ClockSampler(local_rank if gpu_index is None else gpu_index)
    clocks.start()
    start.record(stream)
    for i in range(steps):
        step(i)
    end.record(stream)
    torch.cuda.synchronize()
    clk = clocks.stop()
    if int(status.item()) != 0:
        raise RuntimeError(f"pctree_tree_attention status {int(status.item())}")
    ms = start.elapsed_time(end) / steps
    del q, k, v, ks, vs, out, ws
    torch.cuda.empty_cache()
    nbytes, flops = attention_work(ai)
    peaks, src = measured_peaks()
    hbm = float(peaks["hbm_gbs"])
    tc = float(peaks.get("bf16_tflops", 1900.0))
    gbs = nbytes / (ms * 1e-3) / 1e9
    tfs = flops / (ms * 1e-3) / 1e12
    bound = "hbm" if nbytes / hbm / 1e9 >= flops / tc / 1e12 else "tensor"
    roof = ({"bound": "hbm", "achieved": gbs, "peak": hbm, "unit": "GB/s",
             "frac": gbs / hbm} if bound == "hbm" else
            {"bound": "tensor", "achieved": tfs, "peak": tc, "unit": "TFLOP/s",
             "frac": tfs / tc})
    roof.update({"kernel": "tree_attn_kernel", "peak_source": src,
                 "traffic": None, "other": {"GB/s": gbs, "hbm_frac": gbs / hbm,
                                            "TFLOP/s": tfs, "tensor_frac": tfs / tc}})
    return {
        "metric": "tree-verification attention µs/layer (prefix + ancestors, GQA)",
        "value": ms * 1e3, "unit": "us/layer", "higher_is_better": False,
        "n_gpus": 1, "steps": steps, "warmup": max(warmup, 3),
        "dtype": "bf16", "data": "synthetic (seeded Q/K/V, random breadth-first trees)",
        "config": {"workload": aw.name, "batch": aw.batch, "N": aw.N,
                   "Hq": aw.Hq, "Hkv": aw.Hkv, "D": aw.D,
                   "prefix_max": aw.prefix_max,
                   "mean_prefix": float(ai.prefix_len.mean()),
                   "l2": f"K/V rotated over {n_sets} copies (>= 3x L2)"},
        "bytes_per_layer": nbytes, "flops_per_layer": flops,
        "roofline": roof, "gpu_launches": steps, "clocks": clk}


def run_attention(args, local_rank):
    print(json.dumps(measure_attention(args.attn_workload, local_rank,
                                       args.steps, args.warmup)), flush=True)


def main():
    args = parse_args()
    wl = WORKLOADS[args.workload].with_(mode=args.mode)
    if args.op == "attention":
        run_attention(args, int(os.environ.get("LOCAL_RANK", "0")))
        return
    if args.op == "compact":
        run_compact(args, int(os.environ.get("LOCAL_RANK", "0")))
        return
    if args.sweep:
        run_sweep(args, wl, int(os.environ.get("LOCAL_RANK", "0")))
        return
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))
    if args.impl == "reference":
        run_reference(args, wl, rank, world)
        return
    if world > 1:
        import torch
        import torch.distributed as dist
        torch.cuda.set_device(local_rank)
        dist.init_process_group("nccl")
    try:
        run_ours(args, wl, rank, world, local_rank)
    finally:
        if world > 1:
            import torch.distributed as dist
            dist.destroy_process_group()


if __name__ == "__main__":
    main()
