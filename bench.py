"""Benchmark of the Panther hot path on one or more GB300s (one process per GPU).

    python bench.py [--gpus N] [--steps K] [--warmup W] [--workload scale|batched|small]
                    [--impl ours|reference]

One step is one pass of the Panther hot path over one synthetic graph:
transition tables (Eq. 3) from the device-resident CSR, R random paths
(Algorithm 3), the inverted index (Sec. 3.1), and top-k for every vertex
(Algorithm 1). `value` is whole-job throughput in top-k queries per second
(vertices answered per second, path sampling and indexing included: the
"processing + query" of the paper's Table 2). Multi-GPU runs are independent
replicas (weak scaling): every rank processes its own copy of the workload.

Extra keys: per-stage timings with their roofline fractions, the batched vs
one-launch-per-query comparison on the 1M-vertex batched-query workload, the
oracle timed on a bounded sample on the host cores (`cpu_baseline`), the same
step through the C ABI with host buffers (`e2e`), SM clocks sampled during the
timed region, and the number of library kernel launches in it.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import math
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "paths sampled/s; top-k queries/s batched vs plain at 1 GB300; % of HBM roofline"

# Algorithmic bytes per unit (sector-granular for random accesses):
#   sampler (alias): per step one 32 B sector of the vertex record and one of
#     the alias entry; per path T*64 B + the (T+1)*4 B row  -> 344 B at T=5
#   index: per (vertex, path) pair 4 B key + 4 B id, read + written, per radix
#     pass (3 passes)                                       -> 48 B / pair
#   counting + top-k: per (vertex, path) pair of the index 4 B path id + one
#     32 B path-row sector; per query 8 B*k of output
SAMPLER_B_PER_PATH = lambda T: T * 64 + (T + 1) * 4
#   tables: per vertex the row_ptr entry read (8 B) and the vertex record
#     {start, deg, S} written (16 B); per CSR entry col + w read (8 B) and one
#     table entry written (alias 16 B, prefix {cum, col} 8 B)
TABLES_B = lambda g, mode: g.n * 24 + g.m * (8 + (16 if mode == "alias" else 8))
INDEX_B_PER_PAIR = 48
COUNT_B_PER_PAIR = 36


def _peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(p) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


def _src_hash(*files):
    h = hashlib.sha1()
    for f in files:
        with open(os.path.join(ROOT, "paper_1504_02577_gb300", "csrc", f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:12]


# DRAM traffic of a stage per step (dram__bytes_read.sum + dram__bytes_write.sum
# summed over the stage's launches) from one ncu capture of the 5M-vertex case,
# scaled by the units processed (x10 for the 50M-vertex workload: vertices,
# paths and pairs all grow tenfold); valid only while the stage's sources are
# unchanged (SHA-256 of the files), else reported as null. The capture and its
# command are in profiles/.
NCU_TRAFFIC = {
    "tables": {"bytes_5M": 4335235584, "sources": {
        "paper_1504_02577_gb300/csrc/graph.cu": "ddc27aec9543aed73a9bbb3c95e69ed8d2b2f7726b2d6f8367ca312527138159",
        "paper_1504_02577_gb300/csrc/internal.cuh": "eeaad795871497f38ada3cdb5887cd4102974df9c5128b77b77d089a02da2b07",
    }},
    "sample": {"bytes_5M": 7362045184, "sources": {
        "paper_1504_02577_gb300/csrc/sample.cu": "713f6a3de810b6439cc3f67742685cc10f2bb650aa47df9578a0ce4704370efe",
        "paper_1504_02577_gb300/csrc/internal.cuh": "eeaad795871497f38ada3cdb5887cd4102974df9c5128b77b77d089a02da2b07",
    }},
    "index": {"bytes_5M": 3492788224, "sources": {
        "paper_1504_02577_gb300/csrc/index.cu": "b084c0c673378dfb48f331afd6dbea8bf88226e71da2f275fa676cace242a7bf",
        "paper_1504_02577_gb300/csrc/capi.cu": "a595da3269b103efb8a14db77228ffb4a30178e980ced7d39d500de1a1608e08",
        "paper_1504_02577_gb300/csrc/internal.cuh": "eeaad795871497f38ada3cdb5887cd4102974df9c5128b77b77d089a02da2b07",
    }},
    "topk": {"bytes_5M": 7926624768, "sources": {
        "paper_1504_02577_gb300/csrc/topk.cu": "80d957df35b25bf69dafa94bd333bb988621e8257a5d1125e2fa6ac156c82676",
        "paper_1504_02577_gb300/csrc/internal.cuh": "eeaad795871497f38ada3cdb5887cd4102974df9c5128b77b77d089a02da2b07",
    }},
}


def _traffic(stage, scale):
    t = NCU_TRAFFIC.get(stage)
    if not t:
        return None
    import hashlib
    for f, digest in t["sources"].items():
        try:
            with open(os.path.join(ROOT, f), "rb") as fh:
                if hashlib.sha256(fh.read()).hexdigest() != digest:
                    return None
        except OSError:
            return None
    return int(t["bytes_5M"] * scale)


class Clocks:
    """nvidia-smi sampling of SM clocks and throttle reasons during the timed region."""

    def __init__(self, device: int):
        self.device = device
        self.proc = None
        self.path = None

    def __enter__(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.device}", f"--query-gpu={q}",
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None
        time.sleep(0.3)
        return self

    def __exit__(self, *exc):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()

    def summary(self):
        sm, mx, reasons = [], None, set()
        try:
            for ln in open(self.path):
                f = [x.strip() for x in ln.split(",")]
                if len(f) < 9:
                    continue
                try:
                    sm.append(float(f[1]))
                    mx = float(f[2])
                except ValueError:
                    continue
                for name, val in zip(["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown",
                                      "sw_power_cap"], f[5:9]):
                    if val.lower().startswith("active"):
                        reasons.add(name)
            os.unlink(self.path)
        except Exception:
            pass
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": mx,
                "reasons": sorted(reasons), "samples": len(sm)}


def _dist():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def _barrier(ws):
    if ws > 1:
        import torch.distributed as dist
        dist.barrier()


def _max_over_ranks(x: float, ws: int) -> float:
    if ws == 1:
        return x
    import torch
    import torch.distributed as dist
    dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
    t = torch.tensor([x], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def _sample_size(p):
    import paper_1504_02577_gb300 as pk
    if "R" in p:
        return p["R"]
    return pk.panther_sample_size(p["eps"], p["delta"], p["c"], p["T"])


# ------------------------------------------------------------ our arm ---
def run_ours(args, ws, rank, local):
    import torch
    import synth
    import __graft_entry__
    __graft_entry__.build()
    import paper_1504_02577_gb300 as pk

    torch.cuda.set_device(local)
    MODE = pk.MODE_ALIAS if args.mode == "alias" else pk.MODE_PREFIX
    p = dict(synth.WORKLOADS[args.workload])
    if args.n:
        if "R" in p:
            p["R"] = max(1, p["R"] * args.n // p["n"])
        p["n"] = args.n
    t0 = time.time()
    g = synth.workload_graph(args.workload, n=p["n"])
    gen_s = time.time() - t0
    R, T, k = _sample_size(p), p["T"], p["k"]
    dev = f"cuda:{local}"
    d_rp = torch.from_numpy(g.row_ptr).to(dev)
    d_col = torch.from_numpy(g.col).to(dev)
    d_w = torch.from_numpy(g.w.view(np.int32)).to(dev)
    if args.workload == "batched":
        q_host = synth.query_mix(g, p["q_uniform"], p["q_hub"], seed=1)
    else:
        q_host = np.arange(g.n, dtype=np.int32)
    queries = torch.from_numpy(q_host).to(dev)
    nq = int(q_host.shape[0])

    P = pk.Panther(local)
    ev = lambda: torch.cuda.Event(enable_timing=True)
    stages = ["tables", "sample", "index", "topk"]

    def step(record=None):
        s = P.stream
        e = [ev() for _ in range(5)] if record is not None else None
        if e: e[0].record(s)
        P.build_graph(d_rp, d_col, d_w, MODE)
        if e: e[1].record(s)
        P.sample_paths(args.seed, R, T, MODE)
        if e: e[2].record(s)
        P.build_index()
        if e: e[3].record(s)
        ids, cnt = P.topk(queries, k)
        if e: e[4].record(s)
        if record is not None:
            record.append(e)
        return ids, cnt

    # autotune the batched top-k launch shape on this batch (outside the timed region)
    step()
    shape = P.tune_topk(queries, k)
    for _ in range(args.warmup):
        step()
    P.sync()
    torch.cuda.synchronize()
    _barrier(ws)
    rec = []
    l0 = P.launches()
    with Clocks(local) as clk:
        start, end = ev(), ev()
        torch.cuda.synchronize()
        torch.cuda.nvtx.range_push("timed")   # lets a profiler keep only the timed launches
        start.record(P.stream)
        for _ in range(args.steps):
            last = step(rec)
        end.record(P.stream)
        torch.cuda.synchronize()
        torch.cuda.nvtx.range_pop()
    launches = P.launches() - l0
    P.sync()
    tiers = pk.panther_topk_stats(P.h.ctx)
    # the last timed step's results, for the oracle comparison at the end
    checked = None
    if rank == 0 and ws == 1 and not args.no_extras:
        o_t, p_t = P.index_tensors()
        checked = {"paths": P.paths_tensor().cpu().numpy(), "off": o_t.cpu().numpy(), "pid": p_t.cpu().numpy(),
                   "ids": last[0].cpu().numpy(), "cnt": last[1].cpu().numpy().view(np.uint32)}
        del o_t, p_t
    ms_total = start.elapsed_time(end)
    ms_step = _max_over_ranks(ms_total / args.steps, ws)
    stage_ms = {s: statistics.median(r[i].elapsed_time(r[i + 1]) for r in rec) for i, s in enumerate(stages)}
    _barrier(ws)
    clocks = clk.summary()

    # index size for the algorithmic byte counts
    _, _, _, nnz = pk.panther_index_view(P.h.index)
    peak, peak_kind = _peaks()
    algo = {
        "sample": R * SAMPLER_B_PER_PATH(T),
        "index": nnz * INDEX_B_PER_PAIR,
        "topk": nnz * COUNT_B_PER_PAIR + nq * (16 + 8 * k),
        "tables": TABLES_B(g, args.mode),
    }
    stage_obj = {}
    for s in stages:
        gbs = algo[s] / (stage_ms[s] * 1e-3) / 1e9
        stage_obj[s] = {"ms": round(stage_ms[s], 4), "algo_bytes": int(algo[s]), "achieved_gbs": round(gbs, 1),
                        "frac": round(gbs / peak, 4), "traffic": _traffic(s, g.n / 5_000_000)}
    dom = max(stages, key=lambda s: stage_ms[s])
    kernel_name = {"sample": "sample_kernel (one launch)", "index": "index stage (radix passes)",
                   "topk": "top-k stage (lane, group, team, hub kernels)",
                   "tables": "tables stage (stats and alias kernels)"}[dom]
    traffic = _traffic(dom, g.n / 5_000_000)
    roofline = {"bound": "hbm", "kernel": kernel_name, "achieved": stage_obj[dom]["achieved_gbs"], "peak": peak,
                "peak_kind": peak_kind, "unit": "GB/s", "frac": stage_obj[dom]["frac"],
                "traffic": traffic}

    value = ws * nq / (ms_step * 1e-3)
    out = {
        "metric": METRIC, "value": round(value, 1), "unit": "queries/s", "n_gpus": ws, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": round(ms_step, 3), "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "int32/u64 (integer counts)", "data": "synthetic",
        "config": {"workload": args.workload, "graph": f"Chung-Lu n={g.n} m={g.m} mean_deg={p['mean_deg']} "
                   f"gamma={p['gamma']} weights={p['weights'][0]}[{p['weights'][1]},{p['weights'][2]}] seed=1",
                   "R": R, "T": T, "k": k, "queries": nq, "mode": args.mode, "seed": args.seed,
                   "parallelism": f"replicas{ws}", "l2": "inputs larger than L2 (graph and paths)"},
        "paths_sampled_per_s": round(ws * R / (stage_ms["sample"] * 1e-3), 1),
        "stages": stage_obj,
        "roofline": roofline,
        "gpu_launches": int(launches),
        "clocks": clocks,
        "graph_gen_s": round(gen_s, 2),
        "topk_shape": {"threads": shape[0], "table_slots": shape[1], "ctas_per_sm": shape[2]},
        "topk_tiers": dict(zip(["queries", "lane", "group", "warp", "cta", "hub", "hub_via_buckets",
                                "hub_via_tables", "bucket_overflows", "second_passes"], tiers)),
    }

    # batched vs plain on the 1M-vertex batched-query workload (16,384 queries, top-5)
    if rank == 0 and not args.no_extras and args.workload != "batched":
        out["batched_vs_plain"] = batched_vs_plain(pk, torch, local)

    # serving over the resident state of this workload (paths, index, theta)
    topk_checks = []
    if rank == 0 and not args.no_extras and args.workload == "scale":
        P.vectors(50)
        P.sync()
        sv = serve_measure(pk, P.h.ctx, P.h.index, P.h.paths, P.h.vecs, g.n, local, n_burst=300, n_level=400,
                           levels=(0.95,), n_serial=40)
        topk_checks = sv.pop("_topk_checks")
        out["serving"] = sv
        pk.pantherpp_free_vecs(P.h.vecs)
        P.h.vecs = None

    # the unweighted fast path (t_ij = 1/deg) over the same graph: no table,
    # one column entry per step; same step otherwise
    if not args.no_extras and args.workload == "scale":
        out["unweighted"] = unweighted_block(pk, torch, P, d_rp, d_col, args, R, T, k, queries, nq, peak)

    # end to end through the C ABI with host buffers
    if not args.no_extras:
        out["e2e"] = e2e(pk, torch, P, g, R, T, k, q_host, args, ws)
    P.close()

    # the paper's own operating point on this graph: eps = sqrt(1/|E|)
    if rank == 0 and not args.no_extras and args.workload == "scale":
        out["paper_scale_R"] = paper_scale_block(pk, torch, local, d_rp, d_col, d_w, g, T, k, queries, nq)
    del d_rp, d_col, d_w

    # Panther++ k-NN on its own 10M-vertex workload
    if rank == 0 and not args.no_extras and args.workload == "scale":
        out["knn"] = knn_block(pk, torch, local, args)

    if rank == 0 and ws == 1 and not args.no_extras:
        run = OracleRun(g, R, T, k, queries=q_host, keep_rows=checked is not None)
        step_s, topk_s, F, parts = run.step(seed=1)
        out["cpu_baseline"] = run.describe(step_s, topk_s, F, parts)
        if checked is not None:
            out["parity"] = run.check(checked, q_host)
            del checked
        if topk_checks:   # served top-k rows against the oracle (same seed, R, T)
            ok = True
            for q, kk, ids, cnt in topk_checks:
                rid, rcnt = run.o.topk_many(q, kk, threads=run.threads)
                ok &= bool(np.array_equal(ids, rid) and np.array_equal(cnt, rcnt))
            out["serving"]["topk_requests_checked_vs_oracle"] = len(topk_checks)
            out["serving"]["topk_identical_to_oracle"] = ok
    return out


def paper_scale_block(pk, torch, local, d_rp, d_col, d_w, g, T, k, queries, nq, steps=2, warmup=1):
    """The same step at the paper's sample size for this graph: eps =
    sqrt(1/|E|), delta = 0.1, c = 0.5 (its Implementation Notes), i.e.
    R = ceil(0.5 |E| (log2 C(T,2) + 1 + ln 10)) paths: about 13 times the
    workload's R and about 7.9e9 (vertex, path) pairs in the index."""
    E = g.m // 2
    R = pk.panther_sample_size(math.sqrt(1.0 / E), 0.1, 0.5, T)
    ev = lambda: torch.cuda.Event(enable_timing=True)
    out = {"R": R, "eps": f"sqrt(1/{E})", "delta": 0.1, "c": 0.5}
    try:
        with pk.Panther(local) as P:
            rec = []
            for i in range(warmup + steps):
                e = [ev() for _ in range(5)]
                s = P.stream
                e[0].record(s)
                P.build_graph(d_rp, d_col, d_w, pk.MODE_ALIAS)
                e[1].record(s)
                P.sample_paths(1, R, T, pk.MODE_ALIAS)
                e[2].record(s)
                P.build_index()
                e[3].record(s)
                P.topk(queries, k)
                e[4].record(s)
                P.sync()
                if i >= warmup:
                    rec.append(e)
            torch.cuda.synchronize()
            _, _, _, nnz = pk.panther_index_view(P.h.index)
            st = pk.panther_topk_stats(P.h.ctx)
    except pk.PantherError as ex:
        out["error"] = str(ex)
        return out
    names = ["tables", "sample", "index", "topk"]
    ms = {nm: statistics.median(r[i].elapsed_time(r[i + 1]) for r in rec) for i, nm in enumerate(names)}
    tot = statistics.median(r[0].elapsed_time(r[4]) for r in rec)
    out.update({"index_pairs": int(nnz), "ms_per_step": round(tot, 1), "queries_per_s": round(nq / (tot * 1e-3), 1),
                "paths_sampled_per_s": round(R / (ms["sample"] * 1e-3), 1),
                "stages_ms": {nm: round(v, 2) for nm, v in ms.items()},
                "topk_tiers": dict(zip(["queries", "lane", "group", "warp", "cta", "hub", "hub_via_buckets",
                                        "hub_via_tables", "bucket_overflows", "second_passes"], st))})
    return out


def unweighted_block(pk, torch, P, d_rp, d_col, args, R, T, k, queries, nq, peak, steps=5, warmup=2):
    """The step of the main workload on the same graph read as unweighted
    (Eq. (3) with every weight equal): graph records and a copy of col
    instead of alias tables, one column entry per sampling step."""
    ev = lambda: torch.cuda.Event(enable_timing=True)
    rec = []
    for i in range(warmup + steps):
        e = [ev() for _ in range(5)]
        s = P.stream
        e[0].record(s)
        P.build_graph(d_rp, d_col, None, pk.MODE_UNWEIGHTED)
        e[1].record(s)
        P.sample_paths(args.seed, R, T, pk.MODE_UNWEIGHTED)
        e[2].record(s)
        P.build_index()
        e[3].record(s)
        P.topk(queries, k)
        e[4].record(s)
        if i >= warmup:
            rec.append(e)
    P.sync()
    torch.cuda.synchronize()
    names = ["tables", "sample", "index", "topk"]
    ms = {nm: statistics.median(r[i].elapsed_time(r[i + 1]) for r in rec) for i, nm in enumerate(names)}
    tot = statistics.median(r[0].elapsed_time(r[4]) for r in rec)
    m = int(d_col.shape[0])
    n = int(d_rp.shape[0]) - 1
    tb = n * 24 + m * 12          # row_ptr read + vrec written; col read (validation) + col copied
    return {"ms_per_step": round(tot, 3), "queries_per_s": round(nq / (tot * 1e-3), 1),
            "paths_sampled_per_s": round(R / (ms["sample"] * 1e-3), 1),
            "stages_ms": {nm: round(v, 3) for nm, v in ms.items()},
            "tables_algo_bytes": tb, "tables_frac": round(tb / (ms["tables"] * 1e-3) / 1e9 / peak, 4),
            "note": "same graph, weights ignored (t_ij = 1/deg); paths differ from the weighted run"}


def batched_vs_plain(pk, torch, local):
    import synth
    p = synth.WORKLOADS["batched"]
    g = synth.workload_graph("batched")
    R = pk.panther_sample_size(p["eps"], p["delta"], p["c"], p["T"])
    q = torch.from_numpy(synth.query_mix(g, p["q_uniform"], p["q_hub"], seed=1)).to(f"cuda:{local}")
    res = {}
    with pk.Panther(local) as P:
        P.build_graph(g.row_ptr, g.col, g.w, pk.MODE_ALIAS)
        P.sample_paths(1, R, p["T"], pk.MODE_ALIAS)
        P.build_index()
        res["tuned_shape"] = P.tune_topk(q, p["k"])
        for plain in (False, True):
            reps = 10 if not plain else 2
            for _ in range(2):
                P.topk(q, p["k"], plain=plain)
            P.sync()
            torch.cuda.synchronize()
            s, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            l0 = P.launches()
            s.record(P.stream)
            for _ in range(reps):
                a = P.topk(q, p["k"], plain=plain)
            e.record(P.stream)
            torch.cuda.synchronize()
            ms = s.elapsed_time(e) / reps
            res["plain" if plain else "batched"] = {"ms": round(ms, 4), "queries_per_s": round(q.shape[0] / ms * 1e3, 1),
                                                     "launches_per_call": (P.launches() - l0) // reps}
            if plain:
                pl = a
            else:
                bt = a
        P.sync()
        res["identical"] = bool(torch.equal(pl[0], bt[0]) and torch.equal(pl[1], bt[1]))
    res["speedup"] = round(res["plain"]["ms"] / res["batched"]["ms"], 2)
    res["workload"] = f"Chung-Lu n={g.n} mean_deg=20 gamma=2.3 loguniform[1,1024]; R={R} T=5; 16384 queries; top-5"
    return res


def e2e(pk, torch, P, g, R, T, k, q_host, args, ws):
    """The same step through the C ABI with HOST buffers: CSR in, top-k out."""
    rp = torch.from_numpy(g.row_ptr).pin_memory().numpy()
    col = torch.from_numpy(g.col).pin_memory().numpy()
    w = torch.from_numpy(g.w.view(np.int32)).pin_memory().numpy().view(np.uint32)
    qh = torch.from_numpy(q_host).pin_memory().numpy()
    nq = q_host.shape[0]
    ids = torch.empty((nq, k), dtype=torch.int32).pin_memory().numpy()
    cnt = torch.empty((nq, k), dtype=torch.int32).pin_memory().numpy().view(np.uint32)
    ctx = P.h.ctx

    def step():
        mode = pk.MODE_ALIAS if args.mode == "alias" else pk.MODE_PREFIX
        gh = pk.panther_build_graph(ctx, g.n, g.m, rp, col, w, pk.MEM_HOST, mode)
        ph = pk.panther_sample_paths(ctx, gh, args.seed, R, T, mode)
        ih = pk.panther_build_index(ctx, ph)
        pk.panther_topk(ctx, ih, ph, qh, nq, k, ids, cnt, pk.TOPK_BATCHED | pk.IO_HOST)
        pk.panther_free_index(ih)
        pk.panther_free_paths(ph)
        pk.panther_free_graph(gh)

    steps = max(1, min(args.steps, 3))
    step()
    torch.cuda.synchronize()
    _barrier(ws)
    t0 = time.perf_counter()
    for _ in range(steps):
        step()
    torch.cuda.synchronize()
    dt = _max_over_ranks((time.perf_counter() - t0) / steps, ws)
    h2d = g.row_ptr.nbytes + g.col.nbytes + g.w.nbytes + q_host.nbytes
    d2h = ids.nbytes + cnt.nbytes
    return {"value": round(ws * nq / dt, 1), "unit": "queries/s", "ms_per_step": round(dt * 1e3, 3),
            "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": int(d2h)}


# ---------------------------------------------------------- CPU oracle ---
def _cpu_model():
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for ln in out.splitlines():
            if ln.lower().startswith("model name"):
                return ln.split(":", 1)[1].strip()
    except Exception:
        pass
    import platform
    return platform.processor() or platform.machine()


class OracleRun:
    """The oracle on all host cores over the whole workload (CPU baseline).

    Measured in full, on every core (the all-core driver cuts the independent
    outer loops into ranges; results identical to the single-threaded
    oracle): the alias tables of the whole graph, all R paths and the index of
    all of them. Top-k counting over every vertex is estimated from a
    stratified sample by |P_v| (the index is known, so the strata are exact):
    the H heaviest vertices are timed in full; the next stratum (ranks H to
    65,536) and the rest are timed on uniform samples without replacement.
    Each stratum's wall time is F + c * (queries), F being the fixed cost of
    one all-core call (threads, work arrays), measured on `threads` vertices
    without paths; a sample's (wall - F) scales by N_stratum / sample size,
    since its queries are exchangeable draws from the stratum.
    """

    def __init__(self, g, R, T, k, threads=None, queries=None, keep_rows=False):
        import oracle
        oracle.build()
        self.oracle = oracle
        self.g, self.R, self.T, self.k = g, R, T, k
        self.threads = threads or os.cpu_count() or 1
        th = self.threads
        t0 = time.perf_counter()
        tables = oracle.alias_tables(g, threads=th)
        self.t_tables = time.perf_counter() - t0
        t0 = time.perf_counter()
        self.paths = oracle.sample_paths(g, 1, R, T, oracle.ALIAS, tables=tables, threads=th)
        self.t_paths = time.perf_counter() - t0
        del tables
        t0 = time.perf_counter()
        off, pid = oracle.build_index(g.n, self.paths, threads=th)
        self.t_index = time.perf_counter() - t0
        self.o = oracle.Oracle(g.n, self.paths, off, pid)
        sizes = np.diff(off)
        q = np.arange(g.n, dtype=np.int32) if queries is None else np.asarray(queries, dtype=np.int32)
        self.nq = int(q.shape[0])
        order = q[np.lexsort((np.arange(self.nq), -sizes[q]))]
        self.H = min(256, self.nq)
        self.heavy = np.ascontiguousarray(order[: self.H])
        self.mid = order[self.H: min(65_536, self.nq)]
        self.light = order[min(65_536, self.nq):]
        empty = np.nonzero(sizes == 0)[0][:th].astype(np.int32)
        self.empty = empty if empty.size else order[-th:]
        self.o.topk_many(self.empty, k, threads=th)        # first touch of the driver's memory
        self.keep_rows = keep_rows
        self.rows = {}                                      # oracle rows of every timed query (keep_rows)
        self.t_heavy = self._wall(self.heavy)
        self.nnz = int(off[-1])

    def _wall(self, q):
        t0 = time.perf_counter()
        ids, cnt = self.o.topk_many(q, self.k, threads=self.threads)
        t = time.perf_counter() - t0
        if self.keep_rows:
            self.rows[id(q)] = (np.asarray(q), ids, cnt)
        return t

    def check(self, gpu, queries):
        """The GPU's paths and index (in full) and its top-k rows of every
        query the oracle timed here (the heaviest vertices and both samples)
        against the oracle's; queries[i] is the vertex of output row i."""
        res = {"paths_compared": int(gpu["paths"].shape[0]),
               "paths_identical": bool(np.array_equal(gpu["paths"], self.paths)),
               "index_pairs_compared": int(gpu["pid"].shape[0]),
               "index_identical": bool(np.array_equal(gpu["off"], self.o.off)
                                       and np.array_equal(gpu["pid"], self.o.pid[: gpu["pid"].shape[0]])
                                       and gpu["pid"].shape[0] == self.nnz)}
        row_of = np.full(self.g.n, -1, np.int64)
        row_of[np.asarray(queries)] = np.arange(len(queries))
        n_rows, same = 0, True
        for q, ids, cnt in self.rows.values():
            r = row_of[q]
            keep = r >= 0
            same &= bool(np.array_equal(gpu["ids"][r[keep]], ids[keep])
                         and np.array_equal(gpu["cnt"][r[keep]], cnt[keep]))
            n_rows += int(keep.sum())
        res["topk_rows_compared"] = n_rows
        res["topk_identical"] = same
        res["what"] = ("the last timed step's paths and index in full, and its top-k rows of the queries the "
                       "oracle timed (the heaviest vertices and the uniform samples), against the oracle")
        return res

    def step(self, seed, n_mid=8_192, n_light=524_288):
        """One sampled estimate of the all-vertex top-k time (seconds), plus the parts."""
        rng = np.random.default_rng(seed)
        F = statistics.median(self._wall(self.empty) for _ in range(5))
        est = self.t_heavy
        parts = {}
        for name, pop, ns in (("mid", self.mid, n_mid), ("light", self.light, n_light)):
            if pop.size == 0:
                continue
            smp = pop if pop.size <= ns else rng.choice(pop, size=ns, replace=False)
            w = self._wall(np.ascontiguousarray(smp, dtype=np.int32))
            est += F + max(w - F, 0.0) * (pop.size / smp.size)
            parts[name] = (int(smp.size), int(pop.size), w)
        total = self.t_tables + self.t_paths + self.t_index + est
        return total, est, F, parts

    def describe(self, step_s, topk_s, F, parts):
        return {"value": round(self.nq / step_s, 3), "unit": "queries/s", "cores": self.threads, "kind": "oracle",
                "cpu": _cpu_model(),
                "sample": (f"all {self.threads} host threads; measured in full: alias tables of the whole graph "
                           f"({self.t_tables:.1f} s), all {self.R} paths ({self.t_paths:.1f} s), the index of "
                           f"{self.nnz} pairs ({self.t_index:.1f} s), top-{self.k} of the {self.H} vertices with "
                           f"most paths ({self.t_heavy:.1f} s); top-{self.k} of the other {self.nq - self.H} "
                           f"vertices estimated from uniform samples of two |P_v| strata "
                           + ", ".join(f"{a} of {b} ({w:.2f} s)" for a, b, w in parts.values())
                           + f", each scaled as (wall - {F * 1e3:.1f} ms per call) * stratum/sample"),
                "step_s": round(step_s, 2), "topk_s_estimated": round(topk_s, 2),
                "stages_s": {"tables": round(self.t_tables, 2), "paths": round(self.t_paths, 2),
                             "index": round(self.t_index, 2), "topk": round(topk_s, 2)}}


def run_reference(args, ws, rank):
    """The oracle on the host cores as the reference arm.

    Set-up (once): the all-core oracle over the whole workload (tables, all
    paths, index, heaviest vertices; see OracleRun). Each of the warm-up and
    timed steps re-times the alias tables of the whole graph and a fresh pair
    of stratified query samples (seed = step); paths, index and the heaviest
    vertices keep their set-up times. `value` = vertices answered per second
    of the median step."""
    if rank != 0:
        return None
    import synth
    p = synth.WORKLOADS[args.workload]
    g = synth.workload_graph(args.workload)
    import oracle
    oracle.build()
    R = p["R"] if "R" in p else oracle.sample_size(p["eps"], p["delta"], p["c"], p["T"])
    q = synth.query_mix(g, p["q_uniform"], p["q_hub"], seed=1) if args.workload == "batched" else None
    run = OracleRun(g, R, p["T"], p["k"], queries=q)
    steps = []
    for i in range(args.warmup + args.steps):
        t0 = time.perf_counter()
        run.oracle.alias_tables(g, threads=run.threads)
        run.t_tables = time.perf_counter() - t0
        res = run.step(seed=100 + i)
        if i >= args.warmup:
            steps.append(res)
    steps.sort(key=lambda r: r[0])
    med = steps[len(steps) // 2]
    cb = run.describe(*med)
    v = cb["value"]
    return {"impl": "reference", "metric": METRIC, "value": v, "unit": "queries/s", "n_gpus": ws,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(med[0] * 1e3, 1),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "int32/u64 (integer counts)",
            "data": "synthetic", "config": {"workload": args.workload, "R": R, "T": p["T"], "k": p["k"],
                                            "queries": run.nq},
            "cpu_baseline": cb,
            "e2e": {"value": v, "unit": "queries/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}



# ------------------------------------------------------------ k-NN arm ---
def _peak_tensor():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            d = json.load(f)
        return float(d["bf16_tflops"]), "measured"
    except Exception:
        return 1900.0, "fallback"


KN_ALPHA, KN_BETA = 0.0157, 1.6e-5      # the screen kernel's error-bound constants (see knn.cu)


def screening_error(pk, torch, P, theta, nq=16, seed=5):
    """BF16 screening error of the tensor-core screen against the exact integer
    distance and against an FP64 computation, over every screened pair of nq
    queries (half the vertices with the largest |theta|, half uniform).

    y_hat comes from the kernel itself (pantherpp_debug_screen); the exact
    y = |b|^2 - 2 a.b is formed in int64 from four float64 products of 16-bit
    halves (each exact), the FP64 one as |b|^2 - 2 (a.b) in float64."""
    n, D = theta.shape
    t64 = theta.astype(np.float64)
    norm2 = (theta.astype(np.int64) ** 2).sum(axis=1)
    big = np.argsort(-norm2, kind="stable")[: nq // 2]
    rnd = np.random.default_rng(seed).choice(n, size=nq - big.size, replace=False)
    q = np.concatenate([big, rnd]).astype(np.int32)
    npad = pk.pantherpp_debug_screen(P.h.ctx, P.h.vecs)
    dev = f"cuda:{P.device}"
    y = torch.empty((nq, npad), dtype=torch.float32, device=dev)
    cid = torch.empty(npad, dtype=torch.int32, device=dev)
    pk.pantherpp_debug_screen(P.h.ctx, P.h.vecs, torch.as_tensor(q, device=dev), nq, y, cid)
    y, cid = y.cpu().numpy(), cid.cpu().numpy()
    ok = cid >= 0
    c = cid[ok]
    lo, hi = (theta & 0xFFFF).astype(np.float64), (theta >> 16).astype(np.float64)
    a = theta[q].astype(np.int64)
    exact_rows = (theta.max(axis=1) <= 256)
    res = {"queries": int(nq), "pairs": 0, "max_abs_err_vs_exact": 0.0, "mean_abs_err_vs_exact": 0.0,
           "max_abs_err_vs_fp64": 0.0, "mean_abs_err_vs_fp64": 0.0, "max_err_over_bound": 0.0,
           "exact_pairs_nonzero_err": 0}
    tot_e = tot_f = 0.0
    for i in range(nq):
        ai = a[i]
        alo, ahi = (ai & 0xFFFF).astype(np.float64), (ai >> 16).astype(np.float64)
        # a.b = hi.hi 2^32 + (hi.lo + lo.hi) 2^16 + lo.lo, each dot exact in float64 (< 2^53)
        hh = (hi[c] @ ahi).astype(np.int64)
        mid = (hi[c] @ alo + lo[c] @ ahi).astype(np.int64)
        ll = (lo[c] @ alo).astype(np.int64)
        dot = (hh << 32) + (mid << 16) + ll
        y_exact = norm2[c] - 2 * dot
        y_fp64 = norm2[c].astype(np.float64) - 2.0 * (t64[c] @ ai.astype(np.float64))
        yh = y[i][ok].astype(np.float64)
        e_exact = np.abs(yh - y_exact.astype(np.float64))
        e_fp64 = np.abs(yh - y_fp64)
        bound = (KN_ALPHA * math.sqrt(float(norm2[q[i]])) * np.sqrt(norm2[c].astype(np.float64))
                 + KN_BETA * norm2[c].astype(np.float64) + 1.0) * 1.0001
        res["pairs"] += int(c.size)
        res["max_abs_err_vs_exact"] = max(res["max_abs_err_vs_exact"], float(e_exact.max()))
        res["max_abs_err_vs_fp64"] = max(res["max_abs_err_vs_fp64"], float(e_fp64.max()))
        res["max_err_over_bound"] = max(res["max_err_over_bound"], float((e_exact / bound).max()))
        if exact_rows[q[i]]:
            res["exact_pairs_nonzero_err"] += int((e_exact[exact_rows[c]] != 0).sum())
        tot_e += float(e_exact.sum())
        tot_f += float(e_fp64.sum())
    res["mean_abs_err_vs_exact"] = tot_e / max(res["pairs"], 1)
    res["mean_abs_err_vs_fp64"] = tot_f / max(res["pairs"], 1)
    res["fp64_exact_here"] = bool(float(theta.max()) ** 2 * D < 2.0 ** 53)
    for key in list(res):
        if isinstance(res[key], float):
            res[key] = float(f"{res[key]:.6g}")
    return res


def knn_block(pk, torch, local, args):
    """Panther++ on its 10M-vertex workload (Sec. 3.3): theta for every vertex,
    then the exact top-10 nearest vectors of ALL vertices through the BF16
    tensor-core screen + exact rerank (one call), the FP32 form against the
    BF16 form on a sample of queries (identical results required), and the
    screening error of the tensor-core values."""
    import synth
    p = dict(synth.WORKLOADS["knn"])
    g = synth.workload_graph("knn")
    R, T, D, k = p["R"], p["T"], p["D"], p["k"]
    dev = f"cuda:{local}"
    ev = lambda: torch.cuda.Event(enable_timing=True)
    out = {"workload": f"Chung-Lu n={g.n} m={g.m} mean_deg=20 gamma=2.3 loguniform[1,1024]; R={R} T={T} D={D} "
                       f"k={k}"}
    with pk.Panther(local) as P:
        P.build_graph(torch.from_numpy(g.row_ptr).to(dev), torch.from_numpy(g.col).to(dev),
                      torch.from_numpy(g.w.view(np.int32)).to(dev), pk.MODE_ALIAS)
        P.sample_paths(1, R, T, pk.MODE_ALIAS)
        P.build_index()
        e0, e1 = ev(), ev()
        e0.record(P.stream)
        P.vectors(D)
        e1.record(P.stream)
        P.sync()
        out["vectors_ms"] = round(e0.elapsed_time(e1), 2)
        nsm = torch.cuda.get_device_properties(local).multi_processor_count
        ns = min(g.n, 4 * 128 * nsm)
        qs = torch.from_numpy(synth.uniform_ints(ns, g.n, seed=1, stream=0x71)).to(dev)
        res = {}
        for fp32 in (False, True):
            P.knn(qs[:128], k, fp32=fp32)
            P.sync()
            a, b = ev(), ev()
            a.record(P.stream)
            res[fp32] = P.knn(qs, k, fp32=fp32)
            b.record(P.stream)
            P.sync()
            res[fp32] = res[fp32] + (a.elapsed_time(b),)
        identical = bool(torch.equal(res[False][0], res[True][0]) and torch.equal(res[False][1], res[True][1]))
        out["sample"] = {"queries": ns, "bf16_ms": round(res[False][2], 2), "fp32_ms": round(res[True][2], 2),
                         "speedup_bf16_vs_fp32": round(res[True][2] / res[False][2], 2), "identical": identical}
        s_ids, s_d2 = res[False][0], res[False][1]
        del res
        allq = torch.arange(g.n, dtype=torch.int32, device=dev)
        l0 = P.launches()
        a, b = ev(), ev()
        a.record(P.stream)
        ids, d2 = P.knn(allq, k)
        b.record(P.stream)
        P.sync()
        ms = a.elapsed_time(b)
        launches = P.launches() - l0
        st = pk.pantherpp_knn_stats(P.h.ctx)
        # the rows of the sampled queries equal the sampled run's rows
        sel = qs.long()
        same_rows = bool(torch.equal(ids[sel], s_ids) and torch.equal(d2[sel], s_d2))
        out["all_vertices"] = {"queries": g.n, "ms": round(ms, 1), "queries_per_s": round(g.n / ms * 1e3, 1),
                               "gpu_launches": int(launches), "sample_rows_identical": same_rows,
                               "pairs_screened": st[0], "pairs_reranked": st[1], "shortlist_overflow_queries": st[2],
                               "bf16_exact_rows": st[3]}
        del ids, d2, sel, s_ids, s_d2
        npad = ((g.n + 255) // 256) * 256
        flops = 2.0 * g.n * npad * 64
        peak, kind = _peak_tensor()
        tf = flops / (ms * 1e-3) / 1e12
        out["roofline"] = {"bound": "tensor", "kernel": "screen_kernel (tcgen05 bf16, 128x256x64 tiles)",
                           "achieved": round(tf, 1), "peak": peak, "peak_kind": kind, "unit": "TFLOP/s",
                           "frac": round(tf / peak, 4), "traffic": None,
                           "note": "whole k-NN call (screen + rerank) timed; flops = 2 * n * npad * 64"}
        theta = P.theta_tensor().cpu().numpy().view(np.uint32)
        out["screening_error"] = screening_error(pk, torch, P, theta)
    return out


def run_knn(args, ws, rank, local):
    """Panther++ (Sec. 3.3): theta for every vertex, then exact top-10 nearest
    vectors for a batch of queries against all vertices (BF16 tensor-core
    screening + exact rerank), with the FP32 form timed on the same batch."""
    import torch
    import synth
    import __graft_entry__
    __graft_entry__.build()
    import paper_1504_02577_gb300 as pk

    torch.cuda.set_device(local)
    p = dict(synth.WORKLOADS["knn"])
    if args.n:
        p["R"] = max(1, p["R"] * args.n // p["n"])
        p["n"] = args.n
    g = synth.workload_graph("knn", n=p["n"])
    R, T, D, k = p["R"], p["T"], p["D"], p["k"]
    dev = f"cuda:{local}"
    P = pk.Panther(local)
    ev = lambda: torch.cuda.Event(enable_timing=True)
    P.build_graph(g.row_ptr, g.col, g.w, pk.MODE_ALIAS)
    P.sample_paths(1, R, T, pk.MODE_ALIAS)
    P.build_index()
    e0, e1 = ev(), ev()
    e0.record(P.stream)
    P.vectors(D)
    e1.record(P.stream)
    P.sync()
    vec_ms = e0.elapsed_time(e1)
    nq = min(g.n, 4 * 128 * torch.cuda.get_device_properties(local).multi_processor_count)
    qv = torch.from_numpy(synth.uniform_ints(nq, g.n, seed=1, stream=0x71)).to(dev)
    for _ in range(args.warmup):
        P.knn(qv, k)
    P.sync()
    torch.cuda.synchronize()
    _barrier(ws)
    l0 = P.launches()
    with Clocks(local) as clk:
        s, e = ev(), ev()
        torch.cuda.nvtx.range_push("timed")
        s.record(P.stream)
        for _ in range(args.steps):
            ids, d2 = P.knn(qv, k)
        e.record(P.stream)
        torch.cuda.synchronize()
        torch.cuda.nvtx.range_pop()
    launches = P.launches() - l0
    st = pk.pantherpp_knn_stats(P.h.ctx)
    ms = _max_over_ranks(s.elapsed_time(e) / args.steps, ws)
    # FP32 form on the same batch (one timed run)
    P.knn(qv[:128], k, fp32=True)
    P.sync()
    f0, f1 = ev(), ev()
    f0.record(P.stream)
    fids, fd2 = P.knn(qv, k, fp32=True)
    f1.record(P.stream)
    P.sync()
    fp32_ms = f0.elapsed_time(f1)
    identical = bool(torch.equal(ids, fids) and torch.equal(d2, fd2))
    P.close()
    npad = ((g.n + 255) // 256) * 256
    flops = 2.0 * nq * npad * 64
    peak, kind = _peak_tensor()
    tflops = flops / (ms * 1e-3) / 1e12
    clocks = clk.summary()
    return {
        "metric": METRIC, "value": round(ws * nq / (ms * 1e-3), 1), "unit": "k-NN queries/s", "n_gpus": ws,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(ms, 3), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "bf16 screen (fp32 accum) + uint64 rerank",
        "data": "synthetic",
        "config": {"workload": "knn", "graph": f"Chung-Lu n={g.n} m={g.m} mean_deg=20 gamma=2.3 loguniform[1,1024]",
                   "R": R, "T": T, "D": D, "k": k, "queries": nq, "candidates": g.n,
                   "parallelism": f"replicas{ws}", "l2": "candidate matrix (n x 128 B) larger than L2"},
        "roofline": {"bound": "tensor", "kernel": "screen_kernel (tcgen05 bf16)", "achieved": round(tflops, 1),
                     "peak": peak, "peak_kind": kind, "unit": "TFLOP/s", "frac": round(tflops / peak, 4),
                     "traffic": None},
        "vectors_ms": round(vec_ms, 2),
        "fp32": {"ms": round(fp32_ms, 2), "queries_per_s": round(nq / (fp32_ms * 1e-3), 1),
                 "speedup_bf16": round(fp32_ms / ms, 2), "identical": identical},
        "screen_stats": {"pairs": st[0], "kept_for_rerank": st[1], "overflow_queries": st[2], "exact_rows": st[3]},
        "gpu_launches": int(launches), "clocks": clocks,
    }


# ------------------------------------------------------ parameter sweep ---
def run_sweep(args, ws, rank, local):
    """Throughput against the method's parameters on a 5M-vertex graph of the
    scale workload's shape (the performance side of the paper's T, k and D
    studies: T up to 100, k up to 128, D up to 100; D > 56 runs the exact
    brute force):
    sampler and index against T, top-k against T and k, Panther++ vectors and
    k-NN against D. Each point: one warm-up and the median of 3 (one timed
    run for T >= 50 and k > 64)."""
    import torch
    import synth
    import __graft_entry__
    __graft_entry__.build()
    import paper_1504_02577_gb300 as pk

    torch.cuda.set_device(local)
    n = args.n or 5_000_000
    p = dict(synth.WORKLOADS["scale"])
    R = max(1, p["R"] * n // p["n"])
    g = synth.workload_graph("scale", n=n)
    dev = f"cuda:{local}"
    P = pk.Panther(local)
    P.build_graph(torch.from_numpy(g.row_ptr).to(dev), torch.from_numpy(g.col).to(dev),
                  torch.from_numpy(g.w.view(np.int32)).to(dev), pk.MODE_ALIAS)
    allq = torch.arange(g.n, dtype=torch.int32, device=dev)
    ev = lambda: torch.cuda.Event(enable_timing=True)

    def timed(fn, reps=3):
        fn()
        P.sync()
        ts = []
        for _ in range(reps):
            a, b = ev(), ev()
            a.record(P.stream)
            fn()
            b.record(P.stream)
            torch.cuda.synchronize()
            ts.append(a.elapsed_time(b))
        return statistics.median(ts)

    by_T = []
    for T in (2, 3, 5, 10, 20, 31, 50, 100):
        reps = 3 if T <= 31 else 1
        ms_s = timed(lambda: P.sample_paths(args.seed, R, T, pk.MODE_ALIAS), reps)
        ms_i = timed(lambda: P.build_index(), reps)
        ms_k = timed(lambda: P.topk(allq, 10), reps)
        by_T.append({"T": T, "sample_ms": round(ms_s, 3), "paths_per_s": round(R / ms_s * 1e3, 1),
                     "index_ms": round(ms_i, 3), "topk_ms": round(ms_k, 3),
                     "topk_queries_per_s": round(g.n / ms_k * 1e3, 1)})
    P.sample_paths(args.seed, R, 5, pk.MODE_ALIAS)
    P.build_index()
    by_k = []
    for k in (5, 10, 20, 50, 64, 100, 128):
        ms_k = timed(lambda: P.topk(allq, k), 3 if k <= 64 else 1)
        by_k.append({"k": k, "topk_ms": round(ms_k, 3), "topk_queries_per_s": round(g.n / ms_k * 1e3, 1)})
    by_D = []
    q = torch.randint(0, g.n, (4096,), generator=torch.Generator().manual_seed(3), dtype=torch.int32).to(dev)
    for D in (10, 25, 50, 56, 64, 100):
        ms_v = timed(lambda: P.vectors(D), reps=1)
        ms_n = timed(lambda: P.knn(q, 10), 3 if D <= 56 else 1)
        by_D.append({"D": D, "vectors_ms": round(ms_v, 3), "knn_ms_4096q": round(ms_n, 3),
                     "knn_queries_per_s": round(4096 / ms_n * 1e3, 1)})
    P.close()
    best = max(r["topk_queries_per_s"] for r in by_T)
    return {"metric": METRIC, "value": best, "unit": "queries/s (best top-k point)", "n_gpus": ws, "steps": 3,
            "warmup": 1, "ms_per_step": None, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "int32/u64 (integer counts)", "data": "synthetic",
            "config": {"workload": "sweep", "graph": f"Chung-Lu n={g.n} m={g.m} (scale workload shape)", "R": R,
                       "mode": "alias"},
            "by_T": by_T, "by_k": by_k, "by_D": by_D}


# --------------------------------------------------------- serving arm ---
def _requests(n, count, rng):
    """Mixed requests: 75% top-k (k in {5,10,50}, 1-4,096 vertices, log-uniform
    sizes), 25% k-NN (k = 10, 1-1,024 vertices); query vertices uniform."""
    reqs = []
    for _ in range(count):
        if rng.random() < 0.75:
            kind, k, size = 0, int(rng.choice([5, 10, 50])), int(np.floor(4097 ** rng.random()))
        else:
            kind, k, size = 1, 10, int(np.floor(1025 ** rng.random()))
        size = max(1, size)
        q = rng.integers(0, n, size=size).astype(np.int32)
        reqs.append((kind, q, k))
    return reqs


def serve_measure(pk, ctx, ih, ph, vh, n, device, n_burst=300, n_level=400, levels=(0.5, 0.8, 0.95), n_serial=60,
                  oracle_check=None):
    """Request loop over resident paths, index and Panther++ vectors: capacity
    from a saturating burst, then Poisson arrivals at fractions of it (p50 /
    p99 latency), against the same kind of requests executed one after another
    in the plain form; every 20th request of the last level is compared with
    the same request alone (and, given oracle_check, its top-k rows with the
    oracle's)."""
    import threading
    rng = np.random.default_rng(1)

    def outputs(req):
        kind, q, k = req
        return (np.empty((q.shape[0], k), np.int32),
                np.empty((q.shape[0], k), np.uint32 if kind == 0 else np.uint64))

    def alone(req, plain=False):
        kind, q, k = req
        ids, vals = outputs(req)
        if kind == 0:
            flag = pk.TOPK_PLAIN if plain else pk.TOPK_BATCHED
            pk.panther_topk(ctx, ih, ph, q, q.shape[0], k, ids, vals, flag | pk.IO_HOST)
        else:
            pk.pantherpp_knn(ctx, vh, q, q.shape[0], k, ids, vals, pk.KNN_BF16_SCREEN | pk.IO_HOST)
        return ids, vals

    serial = _requests(n, n_serial, rng)
    alone(serial[0], plain=True)
    t0 = time.perf_counter()
    nq_serial = 0
    for r in serial:
        alone(r, plain=True)
        nq_serial += r[1].shape[0]
    serial_qps = nq_serial / (time.perf_counter() - t0)

    srv = pk.panther_serve_create(device, ih, ph, vh, 8 << 30, 4096, 4)

    def run_stream(reqs, rate):
        outs = [outputs(r) for r in reqs]
        tickets = [None] * len(reqs)
        lat = [None] * len(reqs)
        done = threading.Event()

        def waiter():
            for i in range(len(reqs)):
                while tickets[i] is None:
                    time.sleep(0.0002)
                lat[i] = pk.panther_serve_wait(srv, tickets[i], 600.0)
            done.set()

        th = threading.Thread(target=waiter)
        th.start()
        t_start = time.perf_counter()
        t_next = t_start
        arr = np.random.default_rng(7)
        for i, (kind, q, k) in enumerate(reqs):
            if rate > 0:
                t_next += arr.exponential(1.0 / rate)
                while time.perf_counter() < t_next:
                    time.sleep(0.0001)
            while True:
                try:
                    tickets[i] = pk.panther_serve_submit(srv, kind, q, k, outs[i][0], outs[i][1])
                    break
                except pk.PantherError:
                    time.sleep(0.0005)   # full: retry (admission by budget and slots)
        done.wait()
        th.join()
        wall = time.perf_counter() - t_start
        nq = sum(r[1].shape[0] for r in reqs)
        return outs, np.array(lat), wall, nq

    burst = _requests(n, n_burst, rng)
    _, lat_b, wall_b, nq_b = run_stream(burst, 0)
    cap_rps = len(burst) / wall_b
    res_levels = {}
    check = None
    for frac in levels:
        reqs = _requests(n, n_level, rng)
        outs, lat, wall, nq = run_stream(reqs, frac * cap_rps)
        kinds = np.array([r[0] for r in reqs])
        res_levels[str(frac)] = {"offered_rps": round(frac * cap_rps, 1), "achieved_rps": round(len(reqs) / wall, 1),
                                 "queries_per_s": round(nq / wall, 1),
                                 "p50_ms": round(float(np.percentile(lat, 50)), 3),
                                 "p99_ms": round(float(np.percentile(lat, 99)), 3),
                                 "topk_p50_ms": round(float(np.percentile(lat[kinds == 0], 50)), 3),
                                 "topk_p99_ms": round(float(np.percentile(lat[kinds == 0], 99)), 3),
                                 "knn_p50_ms": round(float(np.percentile(lat[kinds == 1], 50)), 3),
                                 "knn_p99_ms": round(float(np.percentile(lat[kinds == 1], 99)), 3)}
        check = (reqs, outs)
    st = pk.panther_serve_stats(srv)
    pk.panther_serve_destroy(srv)
    reqs, outs = check
    same, n_checked = True, 0
    for i in range(0, len(reqs), 20):
        a_ids, a_vals = alone(reqs[i])
        same &= bool(np.array_equal(a_ids, outs[i][0]) and np.array_equal(a_vals, outs[i][1]))
        n_checked += 1
    top = res_levels[str(levels[-1])]
    out = {"capacity_rps": round(cap_rps, 1), "burst_p50_ms": round(float(np.percentile(lat_b, 50)), 3),
           "burst_p99_ms": round(float(np.percentile(lat_b, 99)), 3), "poisson": res_levels,
           "serial_plain_queries_per_s": round(serial_qps, 1),
           "speedup_vs_serial": round(top["queries_per_s"] / serial_qps, 2),
           "identical_alone_and_mixed": same, "requests_checked_alone": n_checked,
           "mix": "75% top-k k in {5,10,50} 1-4096 vertices log-uniform, 25% k-NN k=10 1-1024 vertices",
           "streams": 4, "mem_budget_gib": 8,
           "server_stats": {"submitted": st[0], "completed": st[1], "batches": st[2],
                            "max_requests_per_batch": st[3], "max_batches_in_flight": st[4], "refused": st[5]}}
    out["_topk_checks"] = [(reqs[i][1], reqs[i][2], outs[i][0], outs[i][1])
                           for i in range(0, len(reqs), 20) if reqs[i][0] == 0]
    return out


def run_serve(args, ws, rank, local):
    """Request loop over the resident graph, paths, index and Panther++ vectors
    of the scale workload (see serve_measure)."""
    import torch
    import synth
    import __graft_entry__
    __graft_entry__.build()
    import paper_1504_02577_gb300 as pk

    torch.cuda.set_device(local)
    p = dict(synth.WORKLOADS["scale"])
    if args.n:
        p["R"] = max(1, p["R"] * args.n // p["n"])
        p["n"] = args.n
    g = synth.workload_graph("scale", n=p["n"])
    ctx = pk.panther_create(local)
    gh = pk.panther_build_graph(ctx, g.n, g.m, g.row_ptr, g.col, g.w, pk.MEM_HOST, pk.MODE_ALIAS)
    ph = pk.panther_sample_paths(ctx, gh, 1, p["R"], p["T"], pk.MODE_ALIAS)
    ih = pk.panther_build_index(ctx, ph)
    vh = pk.pantherpp_vectors(ctx, ih, ph, 50)
    pk.panther_free_graph(gh)
    pk.panther_sync(ctx)
    res = serve_measure(pk, ctx, ih, ph, vh, g.n, local)
    res.pop("_topk_checks")
    pk.pantherpp_free_vecs(vh)
    pk.panther_free_index(ih)
    pk.panther_free_paths(ph)
    pk.panther_destroy(ctx)
    top = res["poisson"]["0.95"]
    out = {
        "metric": METRIC, "value": top["queries_per_s"], "unit": "queries/s (served, 0.95 load)", "n_gpus": ws,
        "steps": 300, "warmup": 0, "ms_per_step": None,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "int32/u64 (integer counts)",
        "data": "synthetic",
        "config": {"workload": "serve", "graph": f"Chung-Lu n={g.n} m={g.m} (scale workload)", "R": p["R"]},
    }
    out.update(res)
    return out

def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--workload", default="scale", choices=["scale", "batched", "small", "knn", "serve", "sweep"])
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-extras", action="store_true", help="skip e2e, cpu baseline and batched-vs-plain")
    ap.add_argument("--n", type=int, default=None,
                    help="vertices (smaller case of the same shape: R scales with n; profiling only)")
    ap.add_argument("--config", type=int, choices=[1, 2, 3, 4, 5], default=None,
                    help="workload by number: 1 small, 2 batched, 3 scale, 4 knn, 5 serve")
    ap.add_argument("--mode", default="alias", choices=["alias", "prefix"],
                    help="neighbour selection of Eq. 3 for the sampler (scale/batched/small workloads)")
    ap.add_argument("--seed", type=int, default=1, help="path seed (scale/batched/small workloads)")
    args = ap.parse_args()
    if args.config:
        args.workload = {1: "small", 2: "batched", 3: "scale", 4: "knn", 5: "serve"}[args.config]
    if args.warmup < 3:
        args.warmup = 3
    ws, rank, local = _dist()
    if args.impl == "reference":
        # the oracle runs on the host: rank 0 alone works and prints, the
        # other ranks exit without work
        out = run_reference(args, ws, rank)
        if out is not None:
            print(json.dumps(out), flush=True)
        return
    if ws > 1:
        import torch
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl", device_id=torch.device(f"cuda:{local}"))
    if args.workload == "knn":
        out = run_knn(args, ws, rank, local)
    elif args.workload == "serve":
        out = run_serve(args, ws, rank, local)
    elif args.workload == "sweep":
        out = run_sweep(args, ws, rank, local)
    else:
        out = run_ours(args, ws, rank, local)
    if rank == 0:
        print(json.dumps(out), flush=True)
    if ws > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
