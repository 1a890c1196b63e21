#!/usr/bin/env python
"""Benchmark of the Fusion staged token-adaptation path on GB300.

A step is one pass of the whole path over one synthetic batch: the DeiT-S
12-block schedule (batch 256, N = 197, d = 384, bf16), merging at every block and
exit-check -> compaction -> pruning at blocks 4, 6, 8 and 10; the survivors of
stage s are the input of stage s+1.  There is no transformer block between
stages, so the L2 cache is flushed (a 512 MB write, untimed) before every stage
and every stage reads its input from HBM, as it would after a real block.

value     images/s per stage: images entering each stage, summed over the step's
          stages and over all ranks, divided by the (max over ranks) sum of the
          stages' CUDA-event times.  A step (flushes, events and stages) is captured
          once as a CUDA graph and replayed, as a serving loop would launch it
          (--eager launches every kernel from the host instead).
roofline  the per-sample kernel (merge + prune + gather), which moves almost all
          bytes: algorithmic bytes / event-timed duration vs the measured HBM copy
          bandwidth.
e2e       the same metric through the public C ABI with host buffers: pinned
          host -> device copy of the step's inputs, the chain, device -> host read
          of the results, all inside the timed region, through runner.Pipeline (two
          buffer slots, each step's input copy overlapping the previous step's kernels).
cpu_baseline  the oracle on the host: one process per core, each on a seeded shard of the
          workload (value, cores), and single-threaded on the whole batch (single_core).
parity    the timed steps' outputs against that single-threaded oracle run: per stage batch
          count, offsets, ids, exit masks and tokens (bf16 bit-exact), with the count of
          decisions whose oracle margin is below 1e-6 (near_ties).
side legs the merge router, the pruning router's scores, the MLP exit head, the
          size-aware attention, one full stage alone, and the schedule with the paper's
          MLP exit heads at blocks 8 and 10 (paper_heads).

--impl reference times the CPU oracle (the only other implementation of the
method here) on the host cores, on a bounded sample of the same workload.
"""
from __future__ import annotations

import argparse
import hashlib
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

METRIC = "images/s per merge→exit→prune stage (DeiT-S, b256); % of HBM roofline"
UNIT = "images/s"
DEFAULT_WORKLOAD = "deit_s_chain12_bf16_b256"
FLUSH_BYTES = 512 << 20


def parse_args():
    ap = argparse.ArgumentParser(description=__doc__, formatter_class=argparse.RawDescriptionHelpFormatter)
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--workload", default=DEFAULT_WORKLOAD)
    ap.add_argument("--e2e-steps", type=int, default=None)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--eager", action="store_true", help="launch every step from the host instead of a CUDA graph")
    return ap.parse_args()


def reduce_over_ranks(time_value, units, world, device):
    """The job's time is the slowest rank's and its work the sum of all ranks' (each rank runs
    its own shard of images; no data crosses ranks)."""
    if world <= 1:
        return float(time_value), float(units)
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(time_value)], dtype=torch.float64, device=device)
    u = torch.tensor([float(units)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    dist.all_reduce(u, op=dist.ReduceOp.SUM)
    return float(t.item()), float(u.item())


def dist_env():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            p = json.load(f)
        return float(p["hbm_gbs"]), "measured"
    except (OSError, KeyError, ValueError):
        return 6800.0, "fallback"


# The translation unit of the per-sample kernel k_image_tc: its source and every header it
# includes.  The recorded DRAM traffic stays valid while none of these changes.
IMAGE_TC_SOURCES = ("paper_2607_02612_gb300/csrc/image_tc.cu", "paper_2607_02612_gb300/csrc/sample.cuh",
                    "paper_2607_02612_gb300/csrc/launch.h", "paper_2607_02612_gb300/csrc/plan.cuh",
                    "paper_2607_02612_gb300/csrc/tc.cuh", "paper_2607_02612_gb300/csrc/common.cuh", "include/fusion.h")


def source_hash() -> str:
    h = hashlib.sha256()
    for f in IMAGE_TC_SOURCES:
        with open(os.path.join(ROOT, f), "rb") as fh:
            h.update(f.encode() + fh.read())
    return h.hexdigest()[:16]


def recorded_traffic(workload: str):
    """DRAM bytes per launch of the per-sample kernel from the committed ncu summary,
    only if it was taken on the current kernel sources."""
    try:
        with open(os.path.join(ROOT, "profiles", "traffic.json")) as f:
            t = json.load(f)
    except (OSError, ValueError):
        return None
    e = t.get(workload)
    if not e or e.get("source_hash") != source_hash():
        return None
    return e


# ---------------------------------------------------------------------------
# clocks during the timed region
# ---------------------------------------------------------------------------
class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.path = None

    def __enter__(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "100"], stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except OSError:
            self.proc = None
        time.sleep(0.3)
        return self

    def __exit__(self, *a):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        if self.proc is None or not self.path:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        with open(self.path) as f:
            for line in f:
                parts = [p.strip() for p in line.split(",")]
                if len(parts) < 9:
                    continue
                try:
                    sm.append(float(parts[1]))
                    smax.append(float(parts[2]))
                except ValueError:
                    continue
                for n, v in zip(names, parts[5:9]):
                    if v.lower().startswith("active"):
                        reasons.add(n)
        os.unlink(self.path)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "samples": len(sm), "reasons": sorted(reasons)}


# ---------------------------------------------------------------------------
# algorithmic bytes (compulsory traffic) of one stage, from its inputs and outputs
# ---------------------------------------------------------------------------
def stage_bytes(spec, dtype, dim, in_off, in_ids, out_off, out_ids, classes, row_ids=False):
    """Algorithmic bytes (first kernel, per-sample kernel) of one stage.  Logits are counted for
    the samples that exit only (the call writes no other row); the input row id of every output
    row only when the caller asked for it (row_ids)."""
    eb = 2 if dtype == "bf16" else 4
    B_in = len(in_off) - 1
    B_out = len(out_off) - 1
    counts_in = np.diff(in_off).astype(np.int64)
    counts_out = np.diff(out_off).astype(np.int64)
    surv = {int(t): j for j, t in enumerate(out_ids)}
    per_out = 8 + (4 if row_ids else 0)                                              # size, score (+ row id)
    first = 0
    if spec.exit:
        n_exit = B_in - B_out                                                        # every sample that leaves exited
        first += B_in * dim * eb + classes * dim * eb + classes * 4 + 2 * dim * eb   # CLS rows, W, b, gamma/beta
        first += n_exit * classes * 4 + B_in * (1 + 4)                               # exited logits, mask, max-prob
    first += (B_in + 1) * 4 + B_in * 8 + B_out * 12 + 4                              # offsets, r/rho, plan outputs
    image = 0
    for i in range(B_in):
        t = int(in_ids[i])
        if t not in surv:
            continue
        n_in = int(counts_in[i])
        n_out = int(counts_out[surv[t]])
        r_eff = min(max(int(spec.r[t]), 0), (n_in - 1) // 2) if spec.merge else 0
        rows_read = n_in if r_eff > 0 else n_out     # all keys (= tokens) are needed to decide a merge
        image += rows_read * dim * eb + n_in * 8 + 16                                # tokens, sizes+scores, scalars
        image += n_out * (dim * eb + per_out)                                       # tokens, size, score (, row id)
    return first, image


# ---------------------------------------------------------------------------
# reference arm: the CPU oracle
# ---------------------------------------------------------------------------
def run_reference(args, world, rank):
    """The oracle as it stands, on the host cores: every step covers the workload's whole batch,
    split into one seeded shard per core (one spawned process each, images are independent)."""
    if rank != 0:
        return 0
    import multiprocessing as mp
    from workloads import make_workload
    w = make_workload(args.workload)
    n = w.batch.batch
    procs = max(1, min(os.cpu_count() or 1, n))
    shard = [n // procs + (1 if k < n % procs else 0) for k in range(procs)]
    ctx = mp.get_context("spawn")
    units = 0
    t_total = 0.0
    with ctx.Pool(procs) as pool:
        pool.map(_oracle_shard, [(args.workload, 1, 1000 + k) for k in range(procs)])   # workers up
        for step in range(args.warmup + args.steps):
            jobs = [(args.workload, shard[k], 3000 + 97 * step + k) for k in range(procs)]
            t0 = time.perf_counter()
            outs = pool.map(_oracle_shard, jobs)
            dt = time.perf_counter() - t0
            if step >= args.warmup:
                t_total += dt
                units += sum(u for u, _ in outs)
    value = units / t_total if t_total > 0 else 0.0
    sample = (f"the whole batch of {n} images per step as {procs} seeded shards of {min(shard)}-{max(shard)} images, "
              f"one process per host core, full {len(w.stages)}-stage schedule each")
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * t_total / max(args.steps, 1),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f64", "data": "synthetic",
            "config": {"workload": args.workload, "batch": n, "sample_batch": n, "shards": procs},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": procs, "kind": "oracle", "sample": sample},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


def _oracle_shard(args):
    """One process's share of the all-cores oracle run: the full schedule on its own seeded
    shard of images of the workload (images are independent; compaction is per shard)."""
    name, batch, seed_offset = args
    import oracle
    from workloads import make_workload
    w = make_workload(name, batch=batch, seed_offset=seed_offset)
    t0 = time.perf_counter()
    res = oracle.chain(w)
    dt = time.perf_counter() - t0
    return batch + sum(int(r["n_out"]) for r in res[:-1]), dt


def cpu_baseline(workload_name: str):
    """The oracle on the host cores: single thread on the whole batch (its results also serve
    the parity check of the bench's own outputs), then one process per core, each on its own
    seeded shard of the same workload, started with spawn before any GPU work.  Returns the
    cpu_baseline entry and the oracle's chain."""
    import multiprocessing as mp
    import oracle
    from workloads import make_workload
    w = make_workload(workload_name)
    n = w.batch.batch
    t0 = time.perf_counter()
    res = oracle.chain(w)
    dt = time.perf_counter() - t0
    units = n + sum(int(r["n_out"]) for r in res[:-1])
    one = {"value": units / dt, "unit": UNIT, "cores": 1,
           "sample": f"all {n} images, one full {len(w.stages)}-stage schedule ({dt:.1f} s)"}
    procs = max(1, os.cpu_count() or 1)
    per = max(1, min(n, 2 * n // procs))   # about two single-thread runs' worth of work in total
    ctx = mp.get_context("spawn")
    with ctx.Pool(procs) as pool:
        pool.map(_oracle_shard, [(workload_name, 1, 1000 + k) for k in range(procs)])   # workers up
        t0 = time.perf_counter()
        outs = pool.map(_oracle_shard, [(workload_name, per, 2000 + k) for k in range(procs)])
        wall = time.perf_counter() - t0
    units_all = sum(u for u, _ in outs)
    entry = {"value": units_all / wall, "unit": UNIT, "cores": procs, "kind": "oracle",
             "sample": f"{procs} processes x {per} images (seeded shards of the workload), full "
                       f"{len(w.stages)}-stage schedule each, {wall:.1f} s wall",
             "single_core": one}
    return entry, res


def parity_vs_oracle(chain, o_outs, dtype, near_tie=1e-6):
    """The bench's own outputs against the oracle's chain on the same inputs, sample by sample
    (matched by original id): exit decisions, and each surviving sample's token rows (bf16
    bit-exact; f32 within 1e-5 of the row's largest magnitude) and sizes.  A sample that
    differs where one of its decisions had an oracle margin below 1e-6 (argmax gap, top-r or
    prune boundary gap, |c - tau|) is counted as a near-tie mismatch and left out of the later
    stages; any other difference is a mismatch.  Decisions below the margin are counted."""
    near = {"argmax": 0, "topr": 0, "prune": 0, "exit": 0}
    near_mismatch, mism, compared = 0, 0, 0
    excluded = set()
    o_in_off = chain.inp.offsets.cpu().numpy()
    o_in_ids = np.arange(len(o_in_off) - 1)
    g_in_ids = o_in_ids
    for s, (g, o) in enumerate(zip(chain.outs, o_outs)):
        ag, tg, pg, eg = (np.asarray(o[k]) for k in ("argmax_gap", "topr_gap", "prune_gap", "exit_gap"))
        near["argmax"] += int(np.sum(ag < near_tie))
        near["topr"] += int(np.sum(tg < near_tie))
        near["prune"] += int(np.sum(pg < near_tie))
        near["exit"] += int(np.sum(eg < near_tie))
        nb = int(g["batch"].item())
        g_off = g["offsets"][:nb + 1].cpu().numpy()
        g_of_id = {int(t): j for j, t in enumerate(g["ids"][:nb].cpu().numpy())}
        g_mask = None
        if g.get("exit_mask") is not None:   # by original id (the GPU's own input order)
            gm = g["exit_mask"].cpu().numpy()
            g_mask = {int(t): int(gm[k]) for k, t in enumerate(g_in_ids)}
        t_g = int(g_off[-1])
        gx = g["x"][:t_g].contiguous()
        gx = gx.view(torch_int16()).cpu().numpy().view(np.uint16) if dtype == "bf16" else gx.float().cpu().numpy()
        gsz = g["sizes"][:t_g].cpu().numpy()
        o_of_id = {int(t): j for j, t in enumerate(o["ids"])}
        for i, t in enumerate(o_in_ids):
            t = int(t)
            if t in excluded:
                continue
            a0, a1 = int(o_in_off[i]), int(o_in_off[i + 1])
            near_i = bool(np.any(ag[a0:a1] < near_tie) or tg[i] < near_tie or pg[i] < near_tie or eg[i] < near_tie)
            ok = (t in o_of_id) == (t in g_of_id)
            if ok and g_mask is not None:
                ok = t in g_mask and int(o["exit_mask"][i]) == g_mask[t]
            if ok and t in o_of_id:
                jo, jg = o_of_id[t], g_of_id[t]
                r0, r1 = int(o["offsets"][jo]), int(o["offsets"][jo + 1])
                q0, q1 = int(g_off[jg]), int(g_off[jg + 1])
                ok = r1 - r0 == q1 - q0 and np.array_equal(gsz[q0:q1], o["sizes"][r0:r1])
                if ok and dtype == "bf16":
                    ok = np.array_equal(gx[q0:q1], o["x"][r0:r1])
                elif ok:
                    ox = np.asarray(o["x"][r0:r1], np.float64)
                    scale = np.maximum(np.abs(ox).max(axis=1, keepdims=True), 1e-30) if r1 > r0 else 1.0
                    ok = bool(np.all(np.abs(gx[q0:q1].astype(np.float64) - ox) <= 1e-5 * scale))
            if ok:
                compared += 1
            elif near_i:
                near_mismatch += 1
                excluded.add(t)
            else:
                mism += 1
                excluded.add(t)
        o_in_off, o_in_ids = np.asarray(o["offsets"]), np.asarray(o["ids"])
        g_in_ids = g["ids"][:nb].cpu().numpy()
    return {"sample_stages_compared": compared, "mismatches": mism, "near_tie_mismatches": near_mismatch,
            "near_ties": near, "rule": "exit decisions and token rows bit-exact (bf16) per sample; decisions "
                                       "with an oracle margin below 1e-6 counted, not excused"}


def per_sample_kernel(b):
    """The per-sample kernel a stage of this batch launches: the tcgen05 kernels for bf16 keys
    whose width is a multiple of 64 (the tiled one once a half holds more than 128 tokens,
    i.e. from 258 tokens), the mma.sync / FFMA kernel otherwise."""
    if b.dtype != "bf16" or b.dim % 64:
        return "k_image"
    return "k_image_tc_tiled" if int(np.diff(b.offsets).max()) >= 258 else "k_image_tc"


def torch_int16():
    import torch
    return torch.int16


def oracle_side_legs(b):
    """The oracle beside each side measurement (router, pruning-router scores, MLP exit head,
    attention): bounded samples of the same inputs, single thread, timed before any GPU work."""
    import oracle
    from workloads import POOL_SPATIAL, f32_to_bf16_bits, make_mlp_head, make_router, make_score_head

    def timed(fn, min_s=0.25):   # seconds per call, repeated until at least min_s in total
        reps, t0 = 0, time.perf_counter()
        while True:
            fn()
            reps += 1
            dt = time.perf_counter() - t0
            if dt >= min_s:
                return dt / reps

    def entry(value, unit, sample):
        return {"value": value, "unit": unit, "cores": 1, "kind": "oracle", "sample": sample}

    out = {}
    rs = make_router(np.random.default_rng(2607), b.dim, b.dtype)
    dt = timed(lambda: oracle.merge_router(b.dtype, b.offsets, b.x, rs.w, rs.beta, rs.tau_tgt, rs.tau_ref))
    out["router"] = entry(b.batch / dt, "images/s", f"all {b.batch} images")
    n = min(64, b.batch)
    rows = int(b.offsets[n])
    sh = make_score_head(np.random.default_rng(2608), b.dim, b.dtype)
    dt = timed(lambda: oracle.token_scores(b.dtype, b.offsets[:n + 1], b.x[:rows], sh.w, sh.b))
    out["pruning_router"] = entry(rows / dt, "tokens/s", f"{n} images, {rows} token rows")
    n = min(32, b.batch)
    rows = int(b.offsets[n])
    mh = make_mlp_head(np.random.default_rng(2609), POOL_SPATIAL, b.dim, 2 * b.dim, 1000, b.dtype)
    dt = timed(lambda: oracle.exit_mlp(b.dtype, b.offsets[:n + 1], b.x[:rows], b.sizes[:rows], mh))
    out["exit_mlp"] = entry(n / dt, "images/s", f"{n} images, SpatialPool head, hidden {2 * b.dim}, 1000 classes")
    n = min(2, b.batch)
    rows = int(b.offsets[n])
    qkv = f32_to_bf16_bits(np.random.default_rng(2610).standard_normal((rows, 3 * 6 * 64), dtype=np.float32))
    dt = timed(lambda: oracle.attention("bf16", b.offsets[:n + 1], qkv, 6, b.sizes[:rows]))
    out["attention"] = entry(n / dt, "images/s", f"{n} images x 6 heads")
    return out


# ---------------------------------------------------------------------------
# our arm
# ---------------------------------------------------------------------------
def main():
    args = parse_args()
    world, rank, local = dist_env()
    if args.impl == "reference":
        return run_reference(args, world, rank)

    import torch
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)

    import paper_2607_02612_gb300 as fz
    from paper_2607_02612_gb300 import runner
    from workloads import make_workload

    fz.build()
    lib = fz.load()
    assert lib is not None

    # cpu baseline first, before any GPU work (its worker processes are spawned, not forked)
    cpu, o_chain = None, None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        cpu, o_chain = cpu_baseline(args.workload)

    w = make_workload(args.workload, seed_offset=rank)
    b = w.batch
    side_cpu = oracle_side_legs(b) if cpu is not None and args.workload == DEFAULT_WORKLOAD else {}
    specs = w.stages
    classes = max([s.head.classes for s in specs if s.head is not None] + [1])
    fus = runner.Fusion(b.batch, classes, dev)
    db = runner.device_batch(b.dtype, b.offsets, b.x, b.keys, b.sizes, b.scores, device=dev)
    cst = []
    for s in specs:
        r = torch.from_numpy(s.r).to(dev) if s.r is not None else None
        rho = torch.from_numpy(s.rho).to(dev) if s.rho is not None else None
        head = runner.head_tensors(s.head, b.dtype, dev) if s.head is not None else None
        flags = ((fz.FUSION_STAGE_MERGE if s.merge else 0) | (fz.FUSION_STAGE_EXIT if s.exit else 0) |
                 (fz.FUSION_STAGE_PRUNE if s.prune else 0))
        cst.append(runner.ChainStage(flags, r, rho, head))
    chain = runner.Chain(fus, db, cst)
    for o in chain.outs:           # row ids are not needed by the next block
        o["keep_idx"] = None
    S = len(cst)
    flush = torch.empty(FLUSH_BYTES, dtype=torch.uint8, device=dev)

    def barrier():
        if world > 1:
            import torch.distributed as dist
            dist.barrier()

    # The timed steps record events at stage boundaries only: an event record between two
    # kernels costs about one completion step (~2 us) of the stream.  The split of an exit
    # stage between its first kernel (the exit check, or the plan kernel of a batch too large
    # for the fused plan) and the per-sample kernel comes from a second graph with a mid event
    # there, replayed as many times after the timed steps.
    has_first = [bool(specs[s].exit) or b.batch > fz.FUSION_FUSED_PLAN_MAX_BATCH for s in range(S)]

    def run_step(evs, split):
        for s in range(S):
            flush.fill_(s & 0xFF)
            e0, e1, e2 = evs[s]
            fz.fusion_profile_next(e0, e1 if (split and has_first[s]) else None, e2)
            chain.run_stage(s)

    mk = lambda: torch.cuda.Event(enable_timing=True)  # noqa: E731
    step_evs = [(mk(), mk(), mk()) for _ in range(S)]
    split_evs = [(mk(), mk(), mk()) for _ in range(S)]
    for trio in step_evs + split_evs:   # create the CUDA events outside any capture
        for e in trio:
            e.record()
    run_step(split_evs, True)   # one eager step: first launches, kernel attributes
    torch.cuda.synchronize()
    st = int(fus.status.item())
    if st != 0:
        raise SystemExit(f"device status {st} ({fz.fusion_status_string(st)})")
    graph = graph_split = None
    if not args.eager:
        # one step (flushes, events, stages) as a CUDA graph: the launch path a serving loop
        # would use; the events are graph nodes and record at every replay
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            run_step(step_evs, False)
        graph_split = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph_split):
            run_step(split_evs, True)
    one = graph.replay if graph is not None else (lambda: run_step(step_evs, False))
    one_split = graph_split.replay if graph_split is not None else (lambda: run_step(split_evs, True))
    for _ in range(args.warmup):
        one()
        one_split()
    torch.cuda.synchronize()

    stage_rows, first_rows, image_rows = [], [], []
    barrier()
    torch.cuda.synchronize()
    with ClockSampler(local) as clk:
        t0 = time.perf_counter()
        for k in range(args.steps):
            one()
            torch.cuda.synchronize()   # the step's events are read before the next replay
            stage_rows.append([t[0].elapsed_time(t[2]) for t in step_evs])
        wall = time.perf_counter() - t0
    barrier()
    for k in range(args.steps):   # the split, after the timed steps
        one_split()
        torch.cuda.synchronize()
        first_rows.append([t[0].elapsed_time(t[1]) if has_first[s] else 0.0 for s, t in enumerate(split_evs)])
        image_rows.append([t[1].elapsed_time(t[2]) if has_first[s] else t[0].elapsed_time(t[2])
                           for s, t in enumerate(split_evs)])
    stage_ms = np.array(stage_rows)
    first_ms = np.array(first_rows)
    image_ms = np.array(image_rows)
    clocks = clk.summary()
    # the outputs of the timed steps against the oracle's chain on the same inputs
    parity = parity_vs_oracle(chain, o_chain, b.dtype) if o_chain is not None else None

    # images entering each stage and algorithmic bytes, from the (deterministic) outputs
    in_off, in_ids = b.offsets, np.arange(b.batch, dtype=np.int32)
    units_step = 0
    bytes_first = bytes_image = 0
    per_stage = []
    for s in range(S):
        o = chain.outs[s]
        nb = int(o["batch"].item())
        out_off = o["offsets"][:nb + 1].cpu().numpy()
        out_ids = o["ids"][:nb].cpu().numpy()
        f1, im = stage_bytes(specs[s], b.dtype, b.dim, in_off, in_ids, out_off, out_ids,
                             specs[s].head.classes if specs[s].head is not None else 0)
        bytes_first += f1
        bytes_image += im
        units_step += len(in_off) - 1
        per_stage.append({"stage": s + 1, "images_in": len(in_off) - 1, "tokens_in": int(in_off[-1]),
                          "ms": float(np.median(stage_ms[:, s])),
                          "ms_p10_p90": [float(np.percentile(stage_ms[:, s], 10)), float(np.percentile(stage_ms[:, s], 90))],
                          "image_kernel_ms": float(np.median(image_ms[:, s])),
                          "image_kernel_bytes": im, "first_kernel_bytes": f1})
        in_off, in_ids = out_off, out_ids

    step_ms = stage_ms.sum(axis=1)
    total_ms = float(step_ms.sum())
    units = units_step * args.steps
    total_ms, units = reduce_over_ranks(total_ms, units, world, dev)
    value = units / (total_ms / 1e3)
    peak, peak_src = peaks()
    img_s = float(image_ms.sum()) / 1e3
    achieved = bytes_image * args.steps / img_s / 1e9
    step_achieved = (bytes_first + bytes_image) * args.steps / (float(stage_ms.sum()) / 1e3) / 1e9
    tr = recorded_traffic(args.workload)
    # the full stages (exit check -> compaction -> prune, blocks 4/6/8/10): images/s and the
    # fraction of the HBM roofline over all their kernels, per the measurement contract
    full = [s for s in range(S) if specs[s].exit]
    full_stats = None
    if full:
        t_full = float(stage_ms[:, full].sum()) / 1e3
        b_full = sum(per_stage[s]["first_kernel_bytes"] + per_stage[s]["image_kernel_bytes"] for s in full) * args.steps
        full_stats = {"stages": [s + 1 for s in full],
                      "images_per_s": sum(per_stage[s]["images_in"] for s in full) * args.steps / t_full,
                      "achieved_gbs": b_full / t_full / 1e9, "frac": b_full / t_full / 1e9 / peak}
    # the side legs are defined on the DeiT-S batch; other workloads time their own schedule only
    side = args.workload == DEFAULT_WORKLOAD
    solo = run_solo_full_stage(args, fz, runner, w, b, dev, flush, peak) if full and side else None
    router = run_router(args, fz, runner, b, dev, flush, peak) if side else None
    scores = run_token_scores(args, fz, runner, b, dev, flush, peak) if side else None
    exit_mlp = run_exit_mlp(args, fz, runner, b, dev, flush, peak) if side else None
    attention = run_attention(args, fz, runner, b, dev, flush, peak) if side else None
    paper_heads = run_paper_heads(args, fz, runner, w, chain, dev, flush) if side else None
    for name, leg in (("router", router), ("pruning_router", scores), ("exit_mlp", exit_mlp), ("attention", attention)):
        if name in side_cpu:
            leg["cpu_oracle"] = side_cpu[name]

    # ---- end to end through the C ABI with host buffers -------------------------------
    e2e = run_e2e(args, fz, runner, chain, b, dev, S, units_step, barrier, world)

    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": total_ms / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": b.dtype, "data": "synthetic",
        "config": {"workload": args.workload, "batch": b.batch, "tokens": int(np.diff(b.offsets).max()),
                   "dim": b.dim, "stages": S, "exit_blocks": list(w.spec.exit_blocks),
                   "l2": "flushed before every stage (512 MB write, untimed)",
                   "timing": ("CUDA events around each stage's kernels, summed; " +
                              ("eager launches" if args.eager else "one step captured as a CUDA graph and replayed") +
                              "; the exit stages' split between their two kernels from a second replay with an "
                              "event between them (not in the timed steps)")},
        "roofline": {"bound": "hbm", "kernel": per_sample_kernel(b) + " (merge + prune + gather)", "achieved": achieved,
                     "peak": peak, "unit": "GB/s", "frac": achieved / peak, "peak_source": peak_src,
                     "traffic": (tr["dram_bytes_per_launch"] if tr else None),
                     "algorithmic_bytes_per_launch": bytes_image / S,
                     "whole_step_frac": step_achieved / peak},
        "cpu_baseline": cpu,
        "parity": parity,
        "e2e": e2e,
        "gpu_launches": sum(1 + int(has_first[s]) for s in range(S)) * args.steps,
        "clocks": clocks,
        "full_stages": full_stats,
        "solo_full_stage": solo,
        "router": router,
        "pruning_router": scores,
        "exit_mlp": exit_mlp,
        "attention": attention,
        "paper_heads": paper_heads,
        "stages": per_stage,
        "kernel_ms_per_step": {"first (exit check or plan)": float(first_ms.sum(axis=1).mean()),
                               "k_image": float(image_ms.sum(axis=1).mean())},
        "wall_s_timed_region": wall,
        "images_per_s_full_schedule": b.batch * world / (total_ms / args.steps / 1e3),
    }
    if rank == 0:
        print(json.dumps(line), flush=True)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()
    return 0


def run_solo_full_stage(args, fz, runner, w, b, dev, flush, peak):
    """One full stage (merge -> exit check -> compaction -> prune) on the N = 197 input batch with
    the first full stage's router outputs and head: the stand-alone stage beside the schedule."""
    import torch
    spec = next(s for s in w.stages if s.exit)
    r = torch.from_numpy(spec.r).to(dev)
    rho = torch.from_numpy(spec.rho).to(dev)
    head = runner.head_tensors(spec.head, b.dtype, dev)
    flags = fz.FUSION_STAGE_MERGE | fz.FUSION_STAGE_EXIT | fz.FUSION_STAGE_PRUNE
    fus = runner.Fusion(b.batch, spec.head.classes, dev)
    db = runner.device_batch(b.dtype, b.offsets, b.x, b.keys, b.sizes, b.scores, device=dev)
    ch = runner.Chain(fus, db, [runner.ChainStage(flags, r, rho, head)])
    ch.outs[0]["keep_idx"] = None   # as in the schedule: the next block needs no row ids
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    for e in ev:
        e.record()

    def one():
        flush.fill_(7)
        fz.fusion_profile_next(ev[0], None, ev[1])
        ch.run_stage(0)

    one()
    torch.cuda.synchronize()
    g = None
    if not args.eager:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            one()
    run = g.replay if g is not None else one
    for _ in range(args.warmup):
        run()
    ms = []
    for _ in range(args.steps):
        run()
        torch.cuda.synchronize()
        ms.append(ev[0].elapsed_time(ev[1]))
    o = ch.outs[0]
    nb = int(o["batch"].item())
    out_off = o["offsets"][:nb + 1].cpu().numpy()
    out_ids = o["ids"][:nb].cpu().numpy()
    f1, im = stage_bytes(spec, b.dtype, b.dim, b.offsets, np.arange(b.batch, dtype=np.int32), out_off, out_ids,
                         spec.head.classes)
    t = float(np.median(ms)) / 1e3
    return {"batch": b.batch, "tokens": int(np.diff(b.offsets).max()), "ms": t * 1e3,
            "ms_p10_p90": [float(np.percentile(ms, 10)), float(np.percentile(ms, 90))],
            "images_per_s": b.batch / t, "achieved_gbs": (f1 + im) / t / 1e9, "frac": (f1 + im) / t / 1e9 / peak}


def run_router(args, fz, runner, b, dev, flush, peak):
    """The merge router with profile scaling (Eq. 4-5) on the step's input batch: one
    dot product per CLS row; bytes = CLS rows + router weight + offsets/ids + r and mt."""
    import torch
    from workloads import make_router
    rs = make_router(np.random.default_rng(2607), b.dim, b.dtype)
    wt = torch.from_numpy(rs.w.view(np.int16).copy() if b.dtype == "bf16" else rs.w.copy()).to(dev)
    fus = runner.Fusion(b.batch, 1, dev)
    db = runner.device_batch(b.dtype, b.offsets, b.x, b.keys, b.sizes, b.scores, device=dev)
    out = dict(r=torch.zeros(b.batch, dtype=torch.int32, device=dev), m=torch.zeros(b.batch, device=dev))
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    for e in ev:
        e.record()

    def one():
        flush.fill_(3)
        fz.fusion_profile_next(ev[0], None, ev[1])
        fus.merge_router(db, wt, rs.beta, rs.tau_tgt, rs.tau_ref, out=out)

    one()
    torch.cuda.synchronize()
    g = None
    if not args.eager:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            one()
    run = g.replay if g is not None else one
    for _ in range(args.warmup):
        run()
    ms = []
    for _ in range(args.steps):
        run()
        torch.cuda.synchronize()
        ms.append(ev[0].elapsed_time(ev[1]))
    eb = 2 if b.dtype == "bf16" else 4
    nbytes = b.batch * (b.dim * eb + 8 + 8) + b.dim * eb
    t = float(np.median(ms)) / 1e3
    return {"batch": b.batch, "ms": t * 1e3, "images_per_s": b.batch / t, "algorithmic_bytes": nbytes,
            "achieved_gbs": nbytes / t / 1e9, "frac": nbytes / t / 1e9 / peak,
            "note": "one CLS dot product per image in double: launch- and latency-bound by design"}


def run_token_scores(args, fz, runner, b, dev, flush, peak):
    """The linear pruning router (Eq. 8) on every token row of the step's input batch, L2
    flushed before each launch; bytes = token rows + one float32 score per row + head weight
    + offsets."""
    import torch
    from workloads import make_score_head
    h = make_score_head(np.random.default_rng(2608), b.dim, b.dtype)
    wt = torch.from_numpy(h.w.view(np.int16).copy() if b.dtype == "bf16" else h.w.copy()).to(dev)
    fus = runner.Fusion(b.batch, 1, dev)
    db = runner.device_batch(b.dtype, b.offsets, b.x, b.keys, b.sizes, b.scores, device=dev)
    out = torch.zeros(db.max_rows, dtype=torch.float32, device=dev)
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    for e in ev:
        e.record()

    def one():
        flush.fill_(3)
        fz.fusion_profile_next(ev[0], None, ev[1])
        fus.token_scores(db, wt, h.b, out=out)

    one()
    torch.cuda.synchronize()
    g = None
    if not args.eager:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            one()
    run = g.replay if g is not None else one
    for _ in range(args.warmup):
        run()
    ms = []
    for _ in range(args.steps):
        run()
        torch.cuda.synchronize()
        ms.append(ev[0].elapsed_time(ev[1]))
    eb = 2 if b.dtype == "bf16" else 4
    rows = int(b.offsets[-1])
    nbytes = rows * (b.dim * eb + 4) + b.dim * eb + (b.batch + 1) * 4
    t = float(np.median(ms)) / 1e3
    return {"kernel": "k_token_scores", "rows": rows, "ms": t * 1e3, "ms_p10_p90": [float(np.percentile(ms, 10)),
            float(np.percentile(ms, 90))], "algorithmic_bytes": nbytes, "achieved_gbs": nbytes / t / 1e9,
            "frac": nbytes / t / 1e9 / peak, "tokens_per_s": rows / t}


def run_paper_heads(args, fz, runner, w, chain, dev, flush):
    """The same schedule with the paper's exit heads (Sec. III-G): the linear head at blocks 4
    and 6, a SpatialPool MLP head at block 8 and a CLS-only MLP head at block 10 (hidden 2d,
    1000 classes) inside the fused stage (fusion_stage_mlp).  Each MLP head's tau is the median
    of its own max_prob over the images entering its block (about half exit), taken once on
    the device before timing.  Timed like the headline: one step as a CUDA graph, L2 flushed
    before every stage, CUDA events around each stage."""
    import torch
    from workloads import POOL_CLS, POOL_SPATIAL, make_mlp_head
    b = w.batch
    specs = w.stages
    exit_idx = [s for s in range(len(specs)) if specs[s].exit]
    if len(exit_idx) < 4:
        return None
    pools = {exit_idx[2]: POOL_SPATIAL, exit_idx[3]: POOL_CLS}
    rng = np.random.default_rng(2611)
    cst = [runner.ChainStage(st.flags, st.r, st.rho, st.head) for st in chain.stages]
    fus = runner.Fusion(b.batch, max(st.head.classes for st in chain.stages if st.head is not None), dev)
    db = runner.device_batch(b.dtype, b.offsets, b.x, b.keys, b.sizes, b.scores, device=dev)
    for si, pool in sorted(pools.items()):
        head = runner.mlp_head_tensors(make_mlp_head(rng, pool, b.dim, 2 * b.dim, 1000, b.dtype), b.dtype, dev)
        cst[si] = runner.ChainStage(chain.stages[si].flags, chain.stages[si].r, chain.stages[si].rho, None, head)
        # tau from the images entering this block, through the stages before it
        probe = runner.Chain(fus, db, cst[:si + 1])
        for s in range(si):
            probe.run_stage(s)
        bin_ = probe.batches[si]
        mp = fus.exit_check_mlp(bin_, head)["max_prob"]
        nb = int(bin_.batch.item()) if bin_.batch is not None else b.batch
        head.tau = float(torch.median(mp[:nb]).item())
    ch = runner.Chain(fus, db, cst)
    for o in ch.outs:
        o["keep_idx"] = None
    S = len(cst)
    mk = lambda: torch.cuda.Event(enable_timing=True)  # noqa: E731
    evs = [(mk(), mk()) for _ in range(S)]
    for e0, e1 in evs:
        e0.record()
        e1.record()

    def step():
        for s in range(S):
            flush.fill_(s & 0xFF)
            fz.fusion_profile_next(evs[s][0], None, evs[s][1])
            ch.run_stage(s)

    step()
    torch.cuda.synchronize()
    if int(fus.status.item()) != 0:
        raise SystemExit(f"device status {int(fus.status.item())} in the paper-heads schedule")
    g = None
    if not args.eager:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            step()
    run = g.replay if g is not None else step
    for _ in range(args.warmup):
        run()
    rows = []
    for _ in range(args.steps):
        run()
        torch.cuda.synchronize()
        rows.append([e0.elapsed_time(e1) for e0, e1 in evs])
    ms = np.median(np.array(rows), axis=0)
    images = [b.batch] + [int(o["batch"].item()) for o in ch.outs[:-1]]
    return {"heads": "linear at blocks 4 and 6, SpatialPool MLP at block 8, CLS-only MLP at block 10 "
                     "(hidden 2d, 1000 classes, tau = median max_prob of each head's input images)",
            "images_per_s": float(sum(images) / (ms.sum() / 1e3)), "ms_per_step": float(ms.sum()),
            "stage_ms": [round(float(v), 4) for v in ms],
            "images_in": images}


def run_exit_mlp(args, fz, runner, b, dev, flush, peak):
    """The exit check with the paper's block-8 exit head (SpatialPool, 2-layer MLP, hidden
    2d, 1000 classes) on the step's input batch, L2 flushed before each call; bytes = token
    rows + sizes (the pool) + both weight matrices + logits and outputs; events split the
    call into pool + first layer and second layer + softmax."""
    import torch
    from workloads import POOL_SPATIAL, make_mlp_head
    head = make_mlp_head(np.random.default_rng(2609), POOL_SPATIAL, b.dim, 2 * b.dim, 1000, b.dtype)
    ht = runner.mlp_head_tensors(head, b.dtype, dev)
    fus = runner.Fusion(b.batch, 1, dev)
    db = runner.device_batch(b.dtype, b.offsets, b.x, b.keys, b.sizes, b.scores, device=dev)
    nbytes_ws = fz.fusion_exit_mlp_workspace_size(b.batch, b.dim, ht.hidden, ht.classes)
    ws = torch.zeros(nbytes_ws, dtype=torch.uint8, device=dev)
    out = dict(mask=torch.zeros(b.batch, dtype=torch.uint8, device=dev),
               logits=torch.zeros((b.batch, ht.classes), device=dev), maxp=torch.zeros(b.batch, device=dev))
    code = fz.FUSION_BF16 if b.dtype == "bf16" else fz.FUSION_F32
    hs = ht.c_struct()
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
    for e in ev:
        e.record()

    def one():
        flush.fill_(3)
        fz.fusion_profile_next(ev[0], ev[1], ev[2])
        fz.check(fz.fusion_exit_check_mlp(code, db.ragged(), db.x, b.dim, db.sizes, hs, out["mask"], out["logits"],
                                          out["maxp"], ws, nbytes_ws, fus.status))

    one()
    torch.cuda.synchronize()
    g = None
    if not args.eager:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            one()
    run = g.replay if g is not None else one
    for _ in range(args.warmup):
        run()
    ms, ms1 = [], []
    for _ in range(args.steps):
        run()
        torch.cuda.synchronize()
        ms.append(ev[0].elapsed_time(ev[2]))
        ms1.append(ev[0].elapsed_time(ev[1]))
    eb = 2 if b.dtype == "bf16" else 4
    rows = int(b.offsets[-1])
    H, C = ht.hidden, ht.classes
    nbytes = rows * (b.dim * eb + 4) + (H * b.dim + C * H) * eb + b.batch * (C * 4 + 5)
    flops = 2.0 * b.batch * (b.dim * H + H * C)
    t = float(np.median(ms)) / 1e3
    return {"kernels": "k_head_pool, k_exit (first layer), k_exit (second layer)", "batch": b.batch, "hidden": H,
            "classes": C, "ms": t * 1e3, "ms_pool_and_first_layer": float(np.median(ms1)),
            "algorithmic_bytes": nbytes, "achieved_gbs": nbytes / t / 1e9, "frac": nbytes / t / 1e9 / peak,
            "tflops": flops / t / 1e12, "images_per_s": b.batch / t}


def run_attention(args, fz, runner, b, dev, flush, peak):
    """Size-aware attention (the block consuming a compacted batch) over the step's input batch:
    DeiT-S heads (6 x 64), random bf16 q, k, v rows, the batch's token sizes, L2 flushed before
    each launch; bytes = qkv read + output written + sizes; FLOPs = 4 N^2 64 per head and sample
    (q k^T and p v).  Reported against both the HBM and the tensor roofline."""
    import torch
    heads = 6
    rng = np.random.default_rng(2610)
    rows = int(b.offsets[-1])
    qkv = torch.from_numpy(rng.standard_normal((rows, 3 * heads * 64), dtype=np.float32)).to(dev).to(torch.bfloat16)
    db = runner.device_batch(b.dtype, b.offsets, b.x, b.keys, b.sizes, b.scores, device=dev)
    fus = runner.Fusion(b.batch, 1, dev)
    out = torch.empty((rows, heads * 64), dtype=torch.bfloat16, device=dev)
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    for e in ev:
        e.record()

    def one():
        flush.fill_(3)
        fz.fusion_profile_next(ev[0], None, ev[1])
        fus.attention(db, qkv, heads, db.sizes, out=out)

    one()
    torch.cuda.synchronize()
    g = None
    if not args.eager:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            one()
    run = g.replay if g is not None else one
    for _ in range(args.warmup):
        run()
    ms = []
    for _ in range(args.steps):
        run()
        torch.cuda.synchronize()
        ms.append(ev[0].elapsed_time(ev[1]))
    n = np.diff(b.offsets).astype(np.float64)
    nbytes = rows * (3 * heads * 64 * 2 + heads * 64 * 2 + 4)
    flops = float(4.0 * 64 * heads * np.sum(n * n))
    t = float(np.median(ms)) / 1e3
    tpeak, tsrc = None, None
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            tpeak, tsrc = float(json.load(f)["bf16_tflops"]), "measured (cuBLAS bf16 burst)"
    except (OSError, ValueError, KeyError):
        tpeak, tsrc = 1900.0, "fallback"
    return {"kernel": "k_attn_tc", "batch": b.batch, "heads": heads, "tokens": rows, "ms": t * 1e3,
            "ms_p10_p90": [float(np.percentile(ms, 10)), float(np.percentile(ms, 90))],
            "algorithmic_bytes": nbytes, "achieved_gbs": nbytes / t / 1e9, "frac_hbm": nbytes / t / 1e9 / peak,
            "tflops": flops / t / 1e12, "frac_tensor": flops / t / 1e12 / tpeak, "tensor_peak_tflops": tpeak,
            "tensor_peak_source": tsrc, "images_per_s": b.batch / t}


def run_e2e(args, fz, runner, chain, b, dev, S, units_step, barrier, world):
    """Host inputs -> device -> chain -> host results, timed together."""
    import torch
    # the two-slot pipeline fills and drains once per timed region: enough steps that the
    # steady state dominates (10 steps read ~7 % below 60 on the DeiT-S schedule)
    steps = args.e2e_steps or max(60, 3 * args.steps)
    db = chain.inp
    host = {
        "x": torch.from_numpy(np.ascontiguousarray(b.x).view(np.int16) if b.dtype == "bf16" else b.x).pin_memory(),
        "sizes": torch.from_numpy(b.sizes).pin_memory(),
        "scores": torch.from_numpy(b.scores).pin_memory(),
        "offsets": torch.from_numpy(b.offsets).pin_memory(),
    }
    dst = {"x": db.x.view(torch.int16) if b.dtype == "bf16" else db.x, "sizes": db.sizes, "scores": db.scores,
           "offsets": db.offsets}
    h2d = sum(t.numel() * t.element_size() for t in host.values())
    d2h_bytes = []
    if args.eager:
        out = chain.host_results()

        def one():
            for k in host:
                dst[k].copy_(host[k], non_blocking=True)
            chain.run()
            res, n = out.fetch()                             # the result's size, then the result
            d2h_bytes.append(n)

        def drain():
            pass
    else:
        # two slots replayed as CUDA graphs; step k's input copy overlaps step k-1's kernels
        pipe = runner.Pipeline(chain)

        def one():
            r = pipe.submit(host)
            if r is not None:
                d2h_bytes.append(r[1])

        def drain():
            r = pipe.finish()
            d2h_bytes.append(r[1])

    for _ in range(3):
        one()
    drain()
    torch.cuda.synchronize()
    barrier()
    t0 = time.perf_counter()
    for _ in range(steps):
        one()
    drain()
    torch.cuda.synchronize()
    dt = time.perf_counter() - t0
    barrier()
    dt, units = reduce_over_ranks(dt, units_step * steps, world, dev)
    return {"value": units / dt, "unit": UNIT, "h2d_bytes_per_step": int(h2d),
            "d2h_bytes_per_step": int(d2h_bytes[-1]), "steps": steps,
            "note": ("pinned host inputs and outputs, C-ABI chain (no L2 flush); " +
                     ("launched eagerly, one step at a time" if args.eager else
                      "two slots replayed as CUDA graphs, each step's input copy overlapping the previous "
                      "step's kernels") + "; the host reads the survivor count, then the results")}


if __name__ == "__main__":
    sys.exit(main())
