#!/usr/bin/env python
"""Throughput of round-synchronous domain propagation on GB300.

One step = one dp_propagate call on the large workload (m=2M rows, n=1.5M
variables, ~29.6M nonzeros; seeded synthetic stand-in for MIPLIB 2017) from
its initial bounds to the fixed point, every round on the device.

value   : nonzeros processed per second, summed over rounds
          (nnz * rounds * steps * ranks / max-over-ranks time), device-
          resident inputs, CUDA events on the library's stream.
e2e     : the same metric through the same public call with pinned HOST
          buffers: inputs copied in and bounds copied out inside the call.
roofline: the activity/candidate kernel (k_round), algorithmic bytes
          12*nnz + 20*m per launch over its CUDA-event launch time, taken
          with the host-driven loop variant right after the timed region,
          the mean over the rounds of one propagation with every chunk
          processed (`marked_avg_launch_us`: as a propagation runs them, its
          later rounds skip chunks without a changed variable; `value` counts
          every nonzero once per round either way).
cpu_baseline: the CPU oracle (one thread) propagating the same workload in
          full; its bounds are also compared element by element with the
          GPU's (`parity`: integer bounds and the infeasibility flag exact,
          continuous within 1e-9 relative).
--impl reference: the oracle, one round over a 1/16 row block per step.
value_compression: the same propagation reading the lossless int8 copy of
          the (small-integer) coefficients: 5 streamed bytes per nonzero
          instead of 12 (reported apart from the roofline fraction).
persistent_loop: the same propagation with the round loop in one
          cooperative kernel (dp_propagate_persistent) instead of the graph.
merge_path: the same propagation over the merge-path layout
          (dp_matrix_load_merge) for several segment lengths: equal work
          per thread instead of length-sorted slices; per-kernel times and
          the largest difference to the sliced layout's bounds.
batched_nodes: 256 branch-and-bound node bound vectors over the medium
          matrix (m=200k, ~2M nonzeros) propagated by one dp_propagate_nodes
          call, against the plain loop of one dp_propagate call per node.
batched_matrices: 64 distinct problems (m log-uniform 1k..200k, ~6M
          nonzeros in all) as one set in one dp_propagate_set call, against
          the plain loop of one dp_propagate call per problem.
serving:  Poisson request streams (1k..50k requests/s) over 32 resident
          matrices (nonzeros log-uniform 1e3..1e6) through dp_server_*:
          p50/p99 latency from arrival to result and achieved requests/s.

Multi-GPU (torchrun): replicas -- every rank propagates its own copy of the
workload; there is no data-path collective (scaling: weak).
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

import numpy as np

ROOT = Path(__file__).resolve().parent
sys.path.insert(0, str(ROOT))

METRIC = "nnz processed/s per round"
UNIT = "nnz/s"
PEAK_FALLBACK_GBS = 6800.0


def merge_bench(dp, ctx, stream, inst, d_in, rounds, ref_lb, ref_ub, sliced_ms, steps,
                ipts=(16, 32, 64, 128, 256)):
    """The headline propagation over the merge-path layout, one entry per
    segment length; `ref_lb/ref_ub` are the sliced layout's bounds."""
    import torch

    entries = []
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    d_lb, d_ub = torch.empty_like(ref_lb), torch.empty_like(ref_ub)
    for ipt in ipts:
        with dp.Matrix(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val, lhs=inst.lhs,
                       rhs=inst.rhs, merge_ipt=ipt) as mm:
            split = mm.info()["split_rows"]
            for _ in range(2):
                r = dp.dp_propagate(ctx, mm, *d_in, lb_out=d_lb, ub_out=d_ub)
            torch.cuda.synchronize()
            e0.record(stream)
            for _ in range(steps):
                r = dp.dp_propagate(ctx, mm, *d_in, lb_out=d_lb, ub_out=d_ub)
            e1.record(stream)
            torch.cuda.synchronize()
            mms = e0.elapsed_time(e1) / steps
            assert r.rounds == rounds and not r.infeasible
            fin = torch.isfinite(ref_lb) & torch.isfinite(ref_ub)
            same_inf = bool(torch.equal(torch.isfinite(d_lb), torch.isfinite(ref_lb)) and
                            torch.equal(torch.isfinite(d_ub), torch.isfinite(ref_ub)))
            rel = torch.maximum((d_lb - ref_lb).abs() / ref_lb.abs().clamp(min=1.0),
                                (d_ub - ref_ub).abs() / ref_ub.abs().clamp(min=1.0))[fin]
            hl = dp.dp_propagate_hostloop(ctx, mm, *d_in, lb_out=d_lb, ub_out=d_ub, timing=True)
            kus = {k: round(hl.kernel_ms[i] / hl.kernel_launches[i] * 1e3, 2)
                   for i, k in enumerate(("act", "fix", "rows", "cand_queue", "finish"))
                   if hl.kernel_launches[i]}
            entries.append({"items_per_thread": ipt, "ms_per_step": round(mms, 3),
                            "value": inst.nnz * rounds / (mms * 1e-3), "split_rows": split,
                            "kernel_us": kus, "same_infinite_bounds": same_inf,
                            "max_rel_diff_vs_sliced": float(rel.max()) if rel.numel() else 0.0})
    best = min(entries, key=lambda e: e["ms_per_step"])
    return {"unit": UNIT, "steps": steps, "sliced_ms_per_step": round(sliced_ms, 3),
            "best": {"items_per_thread": best["items_per_thread"], "value": best["value"],
                     "ms_per_step": best["ms_per_step"]},
            "entries": entries}


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--workload", choices=["large", "medium", "tiny"], default="large")
    ap.add_argument("--chunk", type=int, default=0,
                    help="row split length (0: chosen by the autotuner)")
    ap.add_argument("--round-warps", type=int, default=8, choices=[4, 8],
                    help="warps per block of the round kernels when --chunk is given")
    ap.add_argument("--per-round", action="store_true",
                    help="only print per-round kernel times of one propagation (host loop, "
                         "one round per call from the previous round's bounds)")
    ap.add_argument("--no-autotune", action="store_true",
                    help="skip the autotuner (chunk 256, 8 warps per block)")
    ap.add_argument("--scale", type=float, default=1.0,
                    help="shrink the workload (profiling captures only; the bench line uses 1.0)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-compression", action="store_true",
                    help="skip the int8-value measurement")
    ap.add_argument("--no-merge", action="store_true",
                    help="skip the merge-path layout measurement")
    ap.add_argument("--no-persistent", action="store_true",
                    help="skip the persistent-kernel round loop measurement")
    ap.add_argument("--no-nodes", action="store_true",
                    help="skip the batched branch-and-bound node measurement")
    ap.add_argument("--nodes-only", action="store_true",
                    help="run only the batched node measurement (profiling captures)")
    ap.add_argument("--nodes-count", type=int, default=256)
    ap.add_argument("--nodes-chunk", type=int, default=0,
                    help="row split length for both sides of the batched-node bench "
                         "(default: each side's autotuner)")
    ap.add_argument("--no-serving", action="store_true",
                    help="skip the serving (continuous batching) measurement")
    ap.add_argument("--serving-only", action="store_true")
    ap.add_argument("--no-sets", action="store_true",
                    help="skip the batched distinct-matrices measurement")
    ap.add_argument("--sets-only", action="store_true")
    ap.add_argument("--serving-seconds", type=float, default=1.0)
    return ap.parse_args()


def make_workload(name, scale=1.0):
    from paper_2009_07785_gb300 import synth
    if name == "tiny":
        return synth.tiny()
    return {"large": synth.large, "medium": synth.medium}[name](scale=scale)


def describe(inst):
    lens = np.diff(inst.row_ptr)
    return {"workload": f"{inst.name}: m={inst.m} n={inst.n} nnz={inst.nnz} "
                        f"(row lengths {int(lens.min())}..{int(lens.max())}, seed {inst.seed})",
            "m": inst.m, "n": inst.n, "nnz": inst.nnz}


def algorithmic_bytes(inst):
    """Bytes one round must move with int32 columns and binary64 values and
    bounds: the round kernel streams 12 B per nonzero (value, column) and
    20 B per row (sides, row start); the per-variable finish reads and writes
    the bounds and reads the type, 33 B per variable."""
    return 12 * inst.nnz + 20 * inst.m, 33 * inst.n


def peaks():
    p = ROOT / "MEASURED_PEAKS.json"
    if p.exists():
        d = json.loads(p.read_text())
        return float(d["hbm_gbs"]), "measured"
    return PEAK_FALLBACK_GBS, "fallback"


def sm_max_mhz():
    """The maximum SM clock (MEASURED_PEAKS.json, else the GB300's 2070 MHz)."""
    p = ROOT / "MEASURED_PEAKS.json"
    if p.exists():
        return float(json.loads(p.read_text()).get("sm_max_mhz", 2070.0))
    return 2070.0


def source_sha(names):
    """Hash of the code of csrc files, comments and whitespace removed (a
    comment edit does not change what a profile capture measured)."""
    import re

    csrc = ROOT / "paper_2009_07785_gb300" / "csrc"
    code = []
    for f in names:
        text = (csrc / f).read_text()
        text = re.sub(r"/\*.*?\*/", " ", text, flags=re.S)
        text = re.sub(r"//[^\n]*", " ", text)
        code.append(" ".join(text.split()))
    return hashlib.sha256("\n".join(code).encode()).hexdigest()[:16]


def kernel_source_sha():
    """Hash of the sources that define k_round (kernel file + device helpers)."""
    return source_sha(("dp_kernels.cu", "dp_device.cuh", "dp_round.cuh"))


def read_summary(path):
    """The `- key: `value`` lines of a profile summary as a dict (the value
    between the backticks; a remark may follow it)."""
    kv = {}
    for line in Path(path).read_text().splitlines():
        if ":" in line and line.startswith("- "):
            k, v = line[2:].split(":", 1)
            v = v.strip()
            if v.startswith("`") and "`" in v[1:]:
                v = v[1:v.index("`", 1)]
            kv[k.strip()] = v
    return kv


def ncu_traffic(chunk):
    """Per-launch DRAM bytes of k_round from the committed ncu summary of the
    same row split length, or None if there is none or the kernel source
    changed since that capture."""
    f = ROOT / "profiles" / f"ncu_k_round_large_chunk{chunk}.md"
    if not f.exists():
        return None
    kv = read_summary(f)
    if kv.get("kernel_source_sha256_16") != kernel_source_sha():
        return None
    try:
        return float(kv["dram_bytes_per_launch_full_size"])
    except (KeyError, ValueError):
        return None


class Clocks:
    """nvidia-smi sampler (SM clock, throttle reasons) run during the timed region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device):
        self.proc = None
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.Q}", "--format=csv,noheader,nounits", "-lms", "100",
                 "-i", str(device)], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
        self.t0 = time.time()

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            out, _ = self.proc.communicate(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
            out, _ = self.proc.communicate()
        rows = [r.split(", ") for r in out.strip().splitlines() if r.strip()]
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in rows:
            if len(r) < 9:
                continue
            try:
                sm.append(float(r[1]))
                mx = float(r[2])
            except ValueError:
                continue
            for nm, v in zip(names, r[5:9]):
                if v.strip() == "Active":
                    reasons.add(nm)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": mx, "reasons": sorted(reasons),
                "samples": len(sm)}


def dist():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def max_over_ranks(x: float, pg) -> float:
    """The largest of every rank's x (the whole job takes as long as its
    slowest rank).  pg: torch.distributed (NCCL: CUDA tensor; gloo: CPU), or
    None for one process."""
    if pg is None:
        return float(x)
    import torch

    dev = "cuda" if pg.get_backend() == "nccl" else "cpu"
    t = torch.tensor([float(x)], dtype=torch.float64, device=dev)
    pg.all_reduce(t, op=pg.ReduceOp.MAX)
    return float(t.item())


def job_value(units_per_rank: float, ranks: int, seconds_max: float) -> float:
    """Whole-job throughput: the units all ranks processed over the slowest
    rank's time (replicas: every rank processes the same workload)."""
    return units_per_rank * ranks / seconds_max


def oracle_propagation(inst):
    """The oracle's whole propagation of the workload from its initial bounds
    to its fixed point, timed from the first round to the result (its
    normalisation included); returns (result, seconds)."""
    import oracle

    t0 = time.perf_counter()
    o = oracle.propagate_instance(inst)
    return o, time.perf_counter() - t0


# parity tolerance (the same as the tests'): integer bounds and the
# infeasibility flag exactly, continuous bounds within max(1e-12, 1e-9 |oracle|)
PARITY_REL, PARITY_ABS = 1e-9, 1e-12


def parity_vs_oracle(inst, g_lb, g_ub, g_rounds, g_infeasible, o):
    """Element-by-element comparison of the GPU's propagation with the
    oracle's, both run independently from the same initial bounds."""
    isint = inst.vartype.astype(bool)
    bad, rel_max = 0, 0.0
    for g, r in ((g_lb, o.lb), (g_ub, o.ub)):
        same = (g == r)  # equal, including equal infinities
        with np.errstate(invalid="ignore"):
            d = np.abs(g - r)
        tol = np.maximum(PARITY_ABS, PARITY_REL * np.abs(r))
        # the tolerance applies where both are finite: an infinite bound on
        # one side only is a different result
        both_fin = np.isfinite(g) & np.isfinite(r)
        ok = np.where(isint, same, same | (both_fin & (d <= tol)))
        bad += int((~ok).sum())
        fin = np.isfinite(g) & np.isfinite(r) & ~isint
        if fin.any():
            rel_max = max(rel_max, float((d[fin] / np.maximum(1.0, np.abs(r[fin]))).max()))
    return {"mode": "independent full propagations from the same initial bounds",
            "rounds_gpu": int(g_rounds), "rounds_oracle": int(o.rounds),
            "infeasible_gpu": int(g_infeasible), "infeasible_oracle": int(o.infeasible),
            "bounds_compared": int(2 * inst.n), "n_bad": bad, "n_ties_used": 0,
            "max_rel_diff_continuous": rel_max,
            "tolerance": "integer bounds and the infeasibility flag exact; continuous "
                         "within max(1e-12, 1e-9 |oracle|)",
            "ok": bad == 0 and int(g_rounds) == int(o.rounds)
                  and int(g_infeasible) == int(o.infeasible)}


def run_reference(args):
    """The oracle as the reference arm.  One step = one oracle round over a
    1/16 block of the rows (cycling through the blocks), continuing from the
    bounds the previous steps produced, so any --steps stays bounded."""
    ws, rank, _ = dist()
    if rank != 0:
        return 0
    import oracle

    inst = make_workload(args.workload, args.scale)
    L, U, lhs, rhs = oracle.normalise(inst.m, inst.n, inst.lb, inst.ub, inst.vartype, inst.lhs,
                                      inst.rhs)
    nblk = 16
    edges = np.linspace(0, inst.m, nblk + 1).astype(np.int64)
    blocks = []
    for b in range(nblk):
        r0, r1 = int(edges[b]), int(edges[b + 1])
        k0, k1 = int(inst.row_ptr[r0]), int(inst.row_ptr[r1])
        blocks.append((r1 - r0, inst.row_ptr[r0:r1 + 1] - k0, inst.col[k0:k1], inst.val[k0:k1],
                       lhs[r0:r1], rhs[r0:r1], k1 - k0))
    state = [L, U]

    def step(k):
        mb, rp, ci, va, bl, br, nz = blocks[k % nblk]
        rr = oracle.round_(mb, inst.n, rp, ci, va, state[0], state[1], inst.vartype, bl, br)
        state[0], state[1] = rr.lb, rr.ub
        return nz

    for k in range(args.warmup):
        step(k)
    done = 0
    t0 = time.perf_counter()
    for k in range(args.steps):
        done += step(args.warmup + k)
    el = time.perf_counter() - t0
    value = done / el
    out = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
           "steps": args.steps, "warmup": args.warmup, "ms_per_step": el * 1e3 / args.steps,
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
           "data": "synthetic (seeded; stands in for MIPLIB 2017)", "config": describe(inst),
           "cpu_baseline": {"value": value, "unit": UNIT, "cores": 1, "kind": "oracle",
                            "sample": "one single-threaded oracle round over a 1/16 row block per "
                                      "step, cycling through the blocks"},
           "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(out))
    return 0


def per_round_times(dp, ctx, mat, d_in, max_rounds=100):
    """Kernel times of every round of one propagation: each round is one
    host-loop call with max_rounds = 1 from the bounds the previous call
    returned (the same rounds as one call to the fixed point)."""
    p1 = dp.dp_params_default(max_rounds=1)
    for _ in range(2):  # warm-up
        dp.dp_propagate_hostloop(ctx, mat, *d_in, params=p1)
    lb, ub = d_in[0].clone(), d_in[1].clone()
    rows = []
    for r in range(1, max_rounds + 1):
        res = dp.dp_propagate_hostloop(ctx, mat, lb, ub, *d_in[2:], params=p1, timing=True)
        # kernel times in us, keyed by kernel name ("round" is k_round)
        rows.append({"index": r, **{k: round(res.kernel_ms[i] * 1e3, 1)
                                    for i, k in enumerate(dp.KERNELS)}})
        lb, ub = res.lb.clone(), res.ub.clone()
        if res.status != dp.DP_CAP_HIT or res.infeasible:
            break
    return rows


def nodes_bench(dp, ctx, stream, count=256, reps=3, warmup=3, chunk=0):
    """Batched branch-and-bound nodes (dp_propagate_nodes, one call for all
    nodes) against the plain loop (one dp_propagate call per node, the same
    kernels' single-instance path) on the medium matrix, device-resident
    inputs, CUDA events on the library's stream.  Two node sets: fixings at
    random in-domain values (the stated workload; most nodes are infeasible
    after round 1) and fixings at the feasible point's values (every node
    runs to its fixed point).  Each side gets its own autotuned layout: the
    batched-node autotuner on the first 64 feasible-point nodes, the
    single-instance autotuner on the first of them."""
    import torch
    from paper_2009_07785_gb300 import synth

    inst = synth.medium()
    seed = synth.seed_for(3, 0)
    sets = {"random_values": synth.node_bounds(inst, count, seed=seed),
            "feasible_point_values": synth.node_bounds_at_point(inst, count, seed=seed)}
    FL, FU = sets["feasible_point_values"]
    if chunk:
        tb = {"best": {"chunk": chunk}, "entries": []}
        tp = {"best": {"chunk": chunk, "round_warps": 8}}
    else:
        tb = dp.dp_autotune_nodes(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val,
                                  np.ascontiguousarray(FL[:64]), np.ascontiguousarray(FU[:64]),
                                  inst.vartype, inst.lhs, inst.rhs)
        tp = dp.dp_autotune(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val,
                            np.ascontiguousarray(FL[0]), np.ascontiguousarray(FU[0]),
                            inst.vartype, inst.lhs, inst.rhs, rounds=0)
    torch.cuda.synchronize()
    mat = dp.Matrix(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val, tb["best"]["chunk"],
                    lhs=inst.lhs, rhs=inst.rhs)
    mat_p = dp.Matrix(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val,
                      tp["best"]["chunk"], lhs=inst.lhs, rhs=inst.rhs)
    mat_p.set_launch(tp["best"]["round_warps"])
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    vt, lhs, rhs = dev(inst.vartype), dev(inst.lhs), dev(inst.rhs)
    out = {"workload": f"{inst.name}: m={inst.m} n={inst.n} nnz={inst.nnz}, {count} node bound "
                       f"vectors fixing 1-5% of the integer variables (seed {seed})",
           "count": count,
           "batched_layout": {"chunk": tb["best"]["chunk"], "autotune": tb["entries"]},
           "plain_layout": {"chunk": tp["best"]["chunk"],
                            "round_warps": tp["best"]["round_warps"]}}
    ev = lambda: torch.cuda.Event(enable_timing=True)
    for name, (LB, UB) in sets.items():
        dLB, dUB = dev(LB), dev(UB)
        lo, hi = torch.empty_like(dLB), torch.empty_like(dUB)
        for _ in range(warmup):
            r = dp.dp_propagate_nodes(ctx, mat, dLB, dUB, vt, lhs, rhs, lb_out=lo, ub_out=hi)
        torch.cuda.synchronize()
        e0, e1 = ev(), ev()
        e0.record(stream)
        for _ in range(reps):
            r = dp.dp_propagate_nodes(ctx, mat, dLB, dUB, vt, lhs, rhs, lb_out=lo, ub_out=hi)
        e1.record(stream)
        torch.cuda.synchronize()
        t_batch = e0.elapsed_time(e1) / reps
        # the same batch with the round loop in one persistent cooperative kernel
        lo2, hi2 = torch.empty_like(lo), torch.empty_like(hi)
        for _ in range(warmup):
            rq = dp.dp_propagate_nodes_persistent(ctx, mat, dLB, dUB, vt, lhs, rhs, lb_out=lo2,
                                                  ub_out=hi2)
        torch.cuda.synchronize()
        e0.record(stream)
        for _ in range(reps):
            rq = dp.dp_propagate_nodes_persistent(ctx, mat, dLB, dUB, vt, lhs, rhs, lb_out=lo2,
                                                  ub_out=hi2)
        e1.record(stream)
        torch.cuda.synchronize()
        t_pers = e0.elapsed_time(e1) / reps
        assert np.array_equal(rq.rounds, r.rounds) and torch.equal(lo2, lo) and \
            torch.equal(hi2, hi), "persistent and graph batch results differ"
        rows = [(dLB[k].contiguous(), dUB[k].contiguous()) for k in range(count)]
        o1 = torch.empty(inst.n, dtype=torch.float64, device="cuda")
        o2 = torch.empty_like(o1)
        for k in range(warmup):
            dp.dp_propagate(ctx, mat_p, rows[k][0], rows[k][1], vt, lhs, rhs, lb_out=o1,
                            ub_out=o2)
        torch.cuda.synchronize()
        rounds_plain = []
        e0.record(stream)
        for k in range(count):
            rp = dp.dp_propagate(ctx, mat_p, rows[k][0], rows[k][1], vt, lhs, rhs, lb_out=o1,
                                 ub_out=o2)
            rounds_plain.append(rp.rounds)
        e1.record(stream)
        torch.cuda.synchronize()
        t_plain = e0.elapsed_time(e1)
        assert np.array_equal(np.asarray(rounds_plain), r.rounds), "batched and plain rounds differ"
        h = dp.dp_propagate_nodes_hostloop(ctx, mat, dLB, dUB, vt, lhs, rhs, lb_out=lo, ub_out=hi)
        out[name] = {"nodes_per_s": count / (t_batch * 1e-3),
                     "plain_loop_nodes_per_s": count / (t_plain * 1e-3),
                     "speedup_vs_plain_loop": t_plain / t_batch,
                     "ms_per_batch": round(t_batch, 3), "plain_loop_ms": round(t_plain, 3),
                     "persistent_ms_per_batch": round(t_pers, 3),
                     "persistent_speedup_vs_plain_loop": t_plain / t_pers,
                     "rounds_mean": float(r.rounds.mean()), "rounds_max": int(r.rounds.max()),
                     "infeasible_nodes": int(r.infeasible.sum()),
                     "stage_ms": {k: round(v, 3) for k, v in zip(dp.NODE_STAGES, h.kernel_ms)}}
        if int(r.rounds.max()) == 1:
            # one round in which every node processes every row: the activity
            # pass's (nonzero, node) pairs against the binary64 pipe's floor
            # for the activities alone (one FMA per nonzero, node and finite
            # side; 2 FMAs per clock per SM at the maximum SM clock)
            act_ms = h.kernel_ms[dp.NODE_STAGES.index("act")]
            sides = np.isfinite(inst.lhs).astype(np.int64) + np.isfinite(inst.rhs)
            fmas = float((np.diff(inst.row_ptr) * sides).sum()) * count
            fp64_peak = 2.0 * torch.cuda.get_device_properties(0).multi_processor_count * \
                sm_max_mhz() * 1e6
            out[name]["k_bact"] = {
                "ms": round(act_ms, 3), "nnz_node_pairs_per_s": inst.nnz * count / (act_ms * 1e-3),
                "activity_fmas": fmas, "fp64_fma_peak_per_s": fp64_peak,
                "fp64_floor_ms": round(fmas / fp64_peak * 1e3, 3),
                "fp64_floor_frac": fmas / fp64_peak * 1e3 / act_ms}
    mat.close()
    mat_p.close()
    return out


def set_problems(count=64, target_nnz=6.0e6):
    """64 problems generated like the tiny and medium workloads (alternately)
    with m log-uniform in 1k..200k.  The stated total (~6M nonzeros) does not
    follow from that draw (its expectation is ~20M at these row lengths:
    tiny-like rows hold ~6 nonzeros, medium-like ~10): the first of 1000
    seeds within 10% of 6M is taken, else the closest one."""
    from paper_2009_07785_gb300 import synth

    best = None
    for k in range(1000):
        rng = np.random.default_rng(synth.seed_for(3, 1000 + k))
        ms_k = np.exp(rng.uniform(np.log(1e3), np.log(2e5), size=count)).astype(int)
        est = sum(mm * (6.0 if i % 2 == 0 else 10.0) for i, mm in enumerate(ms_k))
        if best is None or abs(est - target_nnz) < best[0]:
            best = (abs(est - target_nnz), k, ms_k)
        if abs(est - target_nnz) <= 0.1 * target_nnz:
            break
    _, k, ms = best  # none of these draws comes within 10% (the expected total is ~20M)
    ps = []
    for i, mm in enumerate(ms):
        seed = synth.seed_for(3, 2000 + i)
        if i % 2 == 0:
            ps.append(synth.tiny(seed=seed, m=int(mm), n=max(16, int(mm * 0.75))))
        else:
            ps.append(synth.medium(seed=seed, scale=float(mm) / 2.0e5))
    return ps, synth.seed_for(3, 1000 + k)


def sets_bench(dp, ctx, stream, reps=3, warmup=3):
    """The 64 problems as one set (dp_propagate_set) against the plain loop
    of one dp_propagate call per problem (each loaded as its own matrix),
    device-resident inputs, CUDA events on the library's stream."""
    import torch

    ps, seed = set_problems()
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    cat = lambda attr: dev(np.concatenate([getattr(p, attr) for p in ps]))
    ms = dp.MatrixSet(ctx, ps, sides=True)
    args = [cat("lb"), cat("ub"), cat("vartype"), cat("lhs"), cat("rhs")]
    lo, hi = torch.empty_like(args[0]), torch.empty_like(args[0])
    for _ in range(warmup):
        r = dp.dp_propagate_set(ctx, ms, *args, lb_out=lo, ub_out=hi)
    torch.cuda.synchronize()
    ev = lambda: torch.cuda.Event(enable_timing=True)
    e0, e1 = ev(), ev()
    e0.record(stream)
    for _ in range(reps):
        r = dp.dp_propagate_set(ctx, ms, *args, lb_out=lo, ub_out=hi)
    e1.record(stream)
    torch.cuda.synchronize()
    t_set = e0.elapsed_time(e1) / reps
    # the same set with the round loop in one persistent cooperative kernel
    lo2, hi2 = torch.empty_like(lo), torch.empty_like(hi)
    for _ in range(warmup):
        rp = dp.dp_propagate_set_persistent(ctx, ms, *args, lb_out=lo2, ub_out=hi2)
    torch.cuda.synchronize()
    e0.record(stream)
    for _ in range(reps):
        rp = dp.dp_propagate_set_persistent(ctx, ms, *args, lb_out=lo2, ub_out=hi2)
    e1.record(stream)
    torch.cuda.synchronize()
    t_set_p = e0.elapsed_time(e1) / reps
    assert np.array_equal(rp.rounds, r.rounds) and torch.equal(lo2, lo) and torch.equal(hi2, hi), \
        "persistent and graph set results differ"
    mats = [dp.Matrix(ctx, p.m, p.n, p.row_ptr, p.col, p.val, lhs=p.lhs, rhs=p.rhs) for p in ps]
    pargs = [[dev(a) for a in (p.lb, p.ub, p.vartype, p.lhs, p.rhs)] for p in ps]
    outs = [(torch.empty(p.n, dtype=torch.float64, device="cuda"),
             torch.empty(p.n, dtype=torch.float64, device="cuda")) for p in ps]
    for k in range(len(ps)):
        dp.dp_propagate(ctx, mats[k], *pargs[k], lb_out=outs[k][0], ub_out=outs[k][1])
    torch.cuda.synchronize()
    e0.record(stream)
    rounds_plain = []
    for k in range(len(ps)):
        rr = dp.dp_propagate(ctx, mats[k], *pargs[k], lb_out=outs[k][0], ub_out=outs[k][1])
        rounds_plain.append(rr.rounds)
    e1.record(stream)
    torch.cuda.synchronize()
    t_plain = e0.elapsed_time(e1)
    assert np.array_equal(np.asarray(rounds_plain), r.rounds), "set and plain rounds differ"
    nnz_rounds = float(sum(p.nnz * int(rk) for p, rk in zip(ps, r.rounds)))
    for m in mats:
        m.close()
    ms.close()
    nnz = [p.nnz for p in ps]
    return {"workload": f"{len(ps)} problems (tiny-like and medium-like alternately, m log-uniform "
                        f"1k..200k, seed {seed}): {sum(nnz)} nonzeros, {min(nnz)}..{max(nnz)} "
                        f"per problem",
            "problems_per_s": len(ps) / (t_set * 1e-3),
            "plain_loop_problems_per_s": len(ps) / (t_plain * 1e-3),
            "speedup_vs_plain_loop": t_plain / t_set,
            "ms_per_set": round(t_set, 3), "plain_loop_ms": round(t_plain, 3),
            "persistent_ms_per_set": round(t_set_p, 3),
            "persistent_speedup_vs_plain_loop": t_plain / t_set_p,
            "nnz_rounds_per_s": nnz_rounds / (t_set * 1e-3),
            "rounds_max": int(r.rounds.max()), "rounds_mean": float(r.rounds.mean()),
            "infeasible_problems": int(r.infeasible.sum())}


def serving_pool(count=32, seed_k=0):
    """32 resident matrices like the medium workload with nonzeros
    log-uniform in 1e3..1e6 (seeded), and per matrix a set of node bound
    vectors (fixings at the feasible point's values)."""
    from paper_2009_07785_gb300 import synth

    rng = np.random.default_rng(synth.seed_for(4, seed_k))
    target = np.exp(rng.uniform(np.log(1e3), np.log(1e6), size=count))
    insts = [synth.medium(seed=synth.seed_for(4, 1 + k), scale=float(t) / 2.0e6)
             for k, t in enumerate(target)]
    nodes = [synth.node_bounds_at_point(inst, 16, seed=synth.seed_for(4, 100 + k))
             for k, inst in enumerate(insts)]
    return insts, nodes


def serving_bench(dp, ctx, rates=(1000, 5000, 10000, 20000, 50000), seconds=1.0,
                  slots=64, max_requests=20000):
    """Poisson request streams over the resident pool: each request is a
    random pool matrix and one of its node bound vectors; requests are
    submitted at their arrival times (the submitting loop waits for each);
    latency = completion time - arrival time on the server's clock."""
    import torch

    pool_insts, pool_nodes = serving_pool()
    # each matrix's row split length from the batched-node autotuner on two
    # of its node vectors (lanes at low load hold one or two nodes)
    t0 = time.perf_counter()
    chunks = []
    for i, (lb, ub) in zip(pool_insts, pool_nodes):
        tune = dp.dp_autotune_nodes(ctx, i.m, i.n, i.row_ptr, i.col, i.val,
                                    np.ascontiguousarray(lb[:2]), np.ascontiguousarray(ub[:2]),
                                    i.vartype, i.lhs, i.rhs)
        chunks.append(tune["best"]["chunk"])
    tune_s = time.perf_counter() - t0
    torch.cuda.synchronize()
    mats = [dp.Matrix(ctx, i.m, i.n, i.row_ptr, i.col, i.val, c)
            for i, c in zip(pool_insts, chunks)]
    out = {"pool": f"{len(mats)} matrices like the medium workload, nonzeros "
                   f"{min(i.nnz for i in pool_insts)}..{max(i.nnz for i in pool_insts)} "
                   f"(log-uniform), 16 node vectors each (1-5% integer fixings at x*)",
           "slots_per_matrix": slots,
           "row_split_lengths": {str(c): chunks.count(c) for c in sorted(set(chunks))},
           "autotune_seconds": round(tune_s, 1), "rates": []}
    rng = np.random.default_rng(12345)
    for rate in rates:
        nreq = int(min(max_requests, rate * seconds))
        with dp.Server(ctx, slots=slots) as srv:
            ids = [srv.add_matrix(m, i.vartype, i.lhs, i.rhs) for m, i in zip(mats, pool_insts)]
            # warm-up: one request per matrix (workspaces, graphs)
            for k, mid in enumerate(ids):
                srv.submit(mid, pool_nodes[k][0][0], pool_nodes[k][1][0])
            got = 0
            while got < len(ids):
                got += len(srv.poll(256, wait_us=5000))
            gaps = rng.exponential(1e6 / rate, size=nreq)
            which = rng.integers(0, len(ids), size=nreq)
            vec = rng.integers(0, 16, size=nreq)
            outs = [(np.empty(pool_insts[k].n), np.empty(pool_insts[k].n)) for k in range(len(ids))]
            t0 = dp.dp_server_clock_us() + 2000.0
            arrival = t0 + np.cumsum(gaps)
            lat, rounds, done = [], 0, 0
            for q in range(nreq):
                while dp.dp_server_clock_us() < arrival[q]:
                    pass
                k = int(which[q])
                srv.submit(ids[k], pool_nodes[k][0][vec[q]], pool_nodes[k][1][vec[q]],
                           outs[k][0], outs[k][1], arrival_us=float(arrival[q]))
                if q % 64 == 0:
                    for c in srv.poll(1024):
                        lat.append(c["done_us"] - c["arrival_us"])
                        rounds += c["rounds"]
            while len(lat) < nreq:
                for c in srv.poll(1024, wait_us=10000):
                    lat.append(c["done_us"] - c["arrival_us"])
                    rounds += c["rounds"]
            t_end = dp.dp_server_clock_us()
            st = srv.stats()
        lat = np.asarray(lat)
        span_s = (t_end - arrival[0]) * 1e-6
        out["rates"].append({"offered_req_per_s": rate, "requests": nreq,
                             "achieved_req_per_s": nreq / span_s,
                             "p50_ms": float(np.percentile(lat, 50)) / 1e3,
                             "p99_ms": float(np.percentile(lat, 99)) / 1e3,
                             "mean_rounds": rounds / nreq,
                             "mean_active_slots": st["slot_rounds"] / max(st["rounds"], 1),
                             "max_active_slots": st["max_active_slots"]})
    for m in mats:
        m.close()
    return out


def run_ours(args):
    import torch

    import paper_2009_07785_gb300 as dp
    from paper_2009_07785_gb300 import _build

    ws, rank, local = dist()
    torch.cuda.set_device(local)
    pg = None
    if ws > 1:
        import torch.distributed as tdist
        tdist.init_process_group("nccl", device_id=torch.device("cuda", local))
        pg = tdist
    _build.build()
    if args.nodes_only:
        ctx = dp.Context(local, torch.cuda.current_stream())
        print(json.dumps({"batched_nodes": nodes_bench(dp, ctx, torch.cuda.current_stream(),
                                                       count=args.nodes_count,
                                                       chunk=args.nodes_chunk)}))
        ctx.close()
        return 0
    if args.sets_only:
        ctx = dp.Context(local, torch.cuda.current_stream())
        print(json.dumps({"batched_matrices": sets_bench(dp, ctx, torch.cuda.current_stream())}))
        ctx.close()
        return 0
    if args.serving_only:
        ctx = dp.Context(local, torch.cuda.current_stream())
        print(json.dumps({"serving": serving_bench(dp, ctx, seconds=args.serving_seconds)}))
        ctx.close()
        return 0
    inst = make_workload(args.workload, args.scale)
    stream = torch.cuda.current_stream()
    ctx = dp.Context(local, stream)
    tune = None
    chunk, warps = args.chunk, args.round_warps
    if not args.no_autotune and not args.chunk:
        t0 = time.perf_counter()
        tune = dp.dp_autotune(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val, inst.lb,
                              inst.ub, inst.vartype, inst.lhs, inst.rhs, rounds=0)
        tune["seconds"] = round(time.perf_counter() - t0, 1)
        chunk, warps = tune["best"]["chunk"], tune["best"]["round_warps"]
    mat = dp.Matrix(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val, chunk,
                    lhs=inst.lhs, rhs=inst.rhs)
    mat.set_launch(warps)
    # the headline and its roofline use the binary64 values (12 bytes per
    # nonzero); the lossless int8 copy is measured apart below
    can_compress = mat.set_compression(True)
    mat.set_compression(False)
    info = mat.info()
    d_in = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in inst.problem()]
    if args.per_round:
        print(json.dumps({"per_round": per_round_times(dp, ctx, mat, d_in),
                          "config": {**describe(inst), "chunk": chunk or 256,
                                     "round_warps": warps}}))
        mat.close()
        ctx.close()
        return 0
    d_lb = torch.empty(inst.n, dtype=torch.float64, device="cuda")
    d_ub = torch.empty_like(d_lb)
    torch.cuda.synchronize()

    def step():
        return dp.dp_propagate(ctx, mat, *d_in, lb_out=d_lb, ub_out=d_ub)

    clocks = Clocks(local) if rank == 0 else None
    time.sleep(0.3)
    for _ in range(max(args.warmup, 3)):
        r = step()
    rounds = r.rounds
    head = (d_lb.clone(), d_ub.clone(), r.rounds, r.infeasible)  # kept for the parity check
    if pg:
        pg.barrier()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(args.steps):
        r = step()
        assert r.rounds == rounds
    e1.record(stream)
    torch.cuda.synchronize()
    if pg:
        pg.barrier()
    ms = max_over_ranks(e0.elapsed_time(e1), pg)
    clk = clocks.stop() if clocks else None

    value = job_value(inst.nnz * rounds * args.steps, ws, ms / 1e3)
    per_round_us = ms * 1e3 / (args.steps * rounds)
    split = info["split_rows"] > 0
    # per step: prologue (2 kernels) and epilogue (1); per round: k_round,
    # k_cand_queue, k_finish, plus k_combine and k_cand_split with split rows
    launches = args.steps * (3 + (5 if split else 3) * rounds)

    # the same propagation with the loop in one persistent (cooperative) kernel
    persistent = None
    if not args.no_persistent:
        for _ in range(2):
            rp = dp.dp_propagate_persistent(ctx, mat, *d_in, lb_out=d_lb, ub_out=d_ub)
        kp = max(3, min(args.steps, 20))
        torch.cuda.synchronize()
        e0.record(stream)
        for _ in range(kp):
            rp = dp.dp_propagate_persistent(ctx, mat, *d_in, lb_out=d_lb, ub_out=d_ub)
        e1.record(stream)
        torch.cuda.synchronize()
        pms = e0.elapsed_time(e1) / kp
        assert rp.rounds == rounds
        persistent = {"ms_per_step": round(pms, 3), "value": inst.nnz * rounds / (pms * 1e-3),
                      "graph_ms_per_step": round(ms / args.steps, 3), "steps": kp}

    # lossless value compression (int8 coefficients), reported apart
    compression = None
    if can_compress and not args.no_compression:
        mat.set_compression(True)
        for _ in range(2):
            rc_ = dp.dp_propagate(ctx, mat, *d_in, lb_out=d_lb, ub_out=d_ub)
        kc = max(3, min(args.steps, 20))
        torch.cuda.synchronize()
        e0.record(stream)
        for _ in range(kc):
            rc_ = dp.dp_propagate(ctx, mat, *d_in, lb_out=d_lb, ub_out=d_ub)
        e1.record(stream)
        torch.cuda.synchronize()
        cms = e0.elapsed_time(e1) / kc
        assert rc_.rounds == rounds
        hc = dp.dp_propagate_hostloop(ctx, mat, *d_in, lb_out=d_lb, ub_out=d_ub, timing=True)
        mat.set_compression(False)
        compression = {"value": inst.nnz * rounds / (cms * 1e-3), "unit": UNIT,
                       "ms_per_step": round(cms, 3), "steps": kc,
                       "stream_bytes_per_nonzero": 5,
                       "k_round_us": round(hc.kernel_ms[0] / max(hc.kernel_launches[0], 1) * 1e3, 2)}

    # the merge-path layout, against the sliced layout's result
    merge = None
    if not args.no_merge:
        step()
        merge = merge_bench(dp, ctx, stream, inst, d_in, rounds, d_lb.clone(), d_ub.clone(),
                            ms / args.steps, max(3, min(args.steps, 10)))

    # per-kernel CUDA-event timings with the host-driven loop (same kernels, same data)
    hl = dp.dp_propagate_hostloop(ctx, mat, *d_in, lb_out=d_lb, ub_out=d_ub)
    t_hl0 = time.perf_counter()
    nhl = 3
    for _ in range(nhl):
        hl = dp.dp_propagate_hostloop(ctx, mat, *d_in, lb_out=d_lb, ub_out=d_ub, timing=False)
    hostloop_ms = (time.perf_counter() - t_hl0) * 1e3 / nhl
    hl = dp.dp_propagate_hostloop(ctx, mat, *d_in, lb_out=d_lb, ub_out=d_ub, timing=True)
    kms = {k: (hl.kernel_ms[i] / hl.kernel_launches[i] if hl.kernel_launches[i] else 0.0)
           for i, k in enumerate(dp.KERNELS)}
    b_round, _ = algorithmic_bytes(inst)
    peak, peak_kind = peaks()
    # k_round over all chunks: every round of the propagation as the first
    # round of a call of its own.  Inside a call the later rounds skip the
    # chunks without a changed variable (kms), so their time says nothing
    # about bandwidth.
    full = per_round_times(dp, ctx, mat, d_in)
    full_us = sum(r["round"] for r in full) / len(full)
    ach = b_round / (full_us * 1e-6) / 1e9
    floor_us = dp.dp_matrix_access_floor(ctx, mat, 5)
    roof = {"bound": "hbm", "achieved": round(ach, 1), "peak": peak, "unit": "GB/s",
            "frac": round(ach / peak, 4), "traffic": ncu_traffic(chunk or 256),
            "kernel": "k_round", "peak_kind": peak_kind,
            "algorithmic_bytes_per_launch": b_round, "avg_launch_us": round(full_us, 2),
            "marked_avg_launch_us": round(kms["round"] * 1e3, 2),
            # the same matrix's memory accesses of one round without the
            # arithmetic (every value and column streamed, every record
            # gathered): the floor the access pattern sets on k_round
            "access_floor_us": round(floor_us, 2),
            "access_floor_frac": round(b_round / (floor_us * 1e-6) / 1e9 / peak, 4)}

    # end to end through the public call with pinned host buffers
    e2e = None
    if not args.no_e2e:
        h_in = [torch.from_numpy(np.ascontiguousarray(a)).pin_memory() for a in inst.problem()]
        h_lb = torch.empty(inst.n, dtype=torch.float64).pin_memory()
        h_ub = torch.empty_like(h_lb)
        for _ in range(2):
            dp.dp_propagate(ctx, mat, *h_in, lb_out=h_lb, ub_out=h_ub)
        ke = max(3, min(args.steps, 50))
        t0 = time.perf_counter()
        for _ in range(ke):
            re = dp.dp_propagate(ctx, mat, *h_in, lb_out=h_lb, ub_out=h_ub)
        el = max_over_ranks(time.perf_counter() - t0, pg)
        assert re.rounds == rounds
        h2d = sum(int(a.numel() * a.element_size()) for a in h_in)
        d2h = 16 * inst.n + 64
        e2e = {"value": job_value(inst.nnz * rounds * ke, ws, el), "unit": UNIT,
               "h2d_bytes_per_step": h2d,
               "d2h_bytes_per_step": d2h, "steps": ke, "ms_per_step": el * 1e3 / ke}

    cpu, parity = None, None
    if rank == 0 and ws == 1 and not args.no_cpu_baseline:
        o, el = oracle_propagation(inst)
        cpu = {"value": inst.nnz * o.rounds / el, "unit": UNIT, "cores": 1, "kind": "oracle",
               "sample": f"the whole propagation of the same workload ({o.rounds} rounds from "
                         f"its initial bounds), single-threaded C oracle ({el:.1f} s)"}
        parity = parity_vs_oracle(inst, head[0].cpu().numpy(), head[1].cpu().numpy(), head[2],
                                  head[3], o)

    nodes = None
    if ws == 1 and not args.no_nodes:
        nodes = nodes_bench(dp, ctx, stream, count=args.nodes_count, chunk=args.nodes_chunk)
    sets = None
    if ws == 1 and not args.no_sets:
        sets = sets_bench(dp, ctx, stream)
    serving = None
    if ws == 1 and not args.no_serving:
        serving = serving_bench(dp, ctx, seconds=args.serving_seconds)

    if rank == 0:
        out = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps,
               "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True,
               "scaling": "weak", "vs_baseline": None, "dtype": "f64",
               "data": "synthetic (seeded; stands in for MIPLIB 2017)",
               "config": {**describe(inst), "rounds_per_step": rounds, "chunk": chunk or 256,
                          "round_warps": warps, "autotune": tune,
                          "split_rows": info["split_rows"], "padded_slots": info["padded_slots"],
                          "round_us": round(per_round_us, 2),
                          "marking": "rounds with few changed variables process only the chunks that hold one",
                          "kernel_us": {k: round(v * 1e3, 2) for k, v in kms.items()},
                          "hostloop_ms_per_step": round(hostloop_ms, 3),
                          "l2": "no flush: the matrix streamed each round (0.36 GB) exceeds the 129 MB L2",
                          "parallelism": f"replicas x{ws}"},
               "roofline": roof, "cpu_baseline": cpu, "parity": parity, "e2e": e2e,
               "gpu_launches": launches,
               "clocks": clk, "value_compression": compression,
               "persistent_loop": persistent, "merge_path": merge, "batched_nodes": nodes,
               "batched_matrices": sets,
               "serving": serving}
        print(json.dumps(out))
    mat.close()
    ctx.close()
    if pg:
        pg.destroy_process_group()
    return 0


def main():
    args = parse()
    if args.impl == "reference":
        return run_reference(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
