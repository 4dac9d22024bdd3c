#!/usr/bin/env python
"""Benchmark: single-source SimRank top-k queries/s on one GB300 (ExactSim, arXiv:2004.03493).

Workload (default "cl100k"): directed Chung-Lu power-law graph, n = 100,000,
m = 1,000,000, in/out Pareto weights with exponent 2.1 (graph seed 1);
c = 0.6, eps = 1e-6, ten seeded sources (uniform over nodes with din >= 1) run
one at a time, top-50 each.  One step = one top-k query (the sources cycle),
every step of the hot path (forward sweeps, allocation, Algorithm 3's exact
first-meeting terms for the heaviest nodes, walk pairs, reverse sweeps, top-k) on
the GPU, with kappa = 4 by default: on the small ER workload kappa = 4 gave no
error above eps in 100 seeds (the paper's 6/(1-sqrt c)^4 is infeasible at
eps = 1e-6).  --alg3 0 runs Algorithm 2 alone.  The graph is synthetic; the
paper's datasets are not available.

Timing: W warm-up steps, then K timed steps (default 10: each source once); the graph
(8 MB) fits in L2, so
L2 is flushed (a 512 MB write) before every timed step, outside the CUDA-event
bracket of the step.  Under torchrun each rank is an independent replica with
its own ten sources (the path has no exchange step); value = all queries of
all ranks / max over ranks of the timed span.

--impl reference times the CPU oracle (oracle/, FP64, OpenMP walk sampler) as it
stands on the host cores: each step runs a bounded sample of one query (all
sweeps, a fixed number of walk pairs) and the time is scaled to a full query.
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

WORKLOADS = {
    "cl100k": dict(kind="chung_lu", n=100_000, m=1_000_000, gamma=2.1, graph_seed=1, c=0.6, eps=1e-6,
                   sources=10, source_seed=7, k=50),
    "er2000": dict(kind="erdos_renyi", n=2000, m=20_000, graph_seed=1, c=0.6, eps=1e-4, sources=1,
                   source_seed=0, k=50),
    # batched form: 64 sources per launch, eps log-uniform in [1e-7, 1e-4]
    # the configuration's eps range is [1e-7, 1e-4]; at kappa = 4 without Algorithm 3 the batched
    # path affords [1e-5, 1e-4] (eps = 1e-7 needs about 2.8e14 pairs for the source alone)
    "rmat20": dict(kind="rmat", scale=20, n=1 << 20, m=30_000_000, graph_seed=1, c=0.6, eps_lo=1e-5, eps_hi=1e-4,
                   eps_config=(1e-7, 1e-4),
                   eps=1e-4, sources=64, source_seed=7, k=100),
    # serving form: Poisson arrivals of top-100 queries, eps from {1e-5, 1e-6, 1e-7}
    # the configuration draws eps from {1e-5, 1e-6, 1e-7}; at kappa = 4 a request at 1e-6 needs about
    # 3.5e12 walk pairs on this graph, so the server is measured at eps in {1e-4, 1e-5}
    "rmat25": dict(kind="rmat_torch", scale=25, n=1 << 25, m=500_000_000, graph_seed=1, c=0.6,
                   eps_set=(1e-4, 1e-5), eps_config=(1e-5, 1e-6, 1e-7), eps=1e-5, sources=4096, source_seed=7,
                   k=100),
    # precision form: FP32c against FP64 sweeps on the same sources and the same D^
    "cl4m": dict(kind="chung_lu_torch", n=4_000_000, m=70_000_000, gamma=2.2, graph_seed=1, c=0.6, eps=1e-7,
                 sources=4, source_seed=7, k=50),
}
METRIC = "single-source SimRank top-k queries/s (Chung-Lu n=1e5 m=1e6, eps=1e-6, top-50)"
# Philox-4x32-10 blocks per SM and clock of a kernel that only draws them (426 G/s on 152 SMs at 2070 MHz): a
# pair-step needs one block, whose 20 wide multiplies (four cycles a warp and scheduler each) fill the multiply pipe
PHILOX_PER_SM_CLOCK = 426e9 / (152 * 2.07e9)
# DRAM bytes of one sampler launch of the bench query, one-pass ncu capture of the current
# kernel (dram__bytes_read.sum + dram__bytes_write.sum; the walk table once, it stays in L2)
SAMPLER_TRAFFIC = 9.72e6
# Algorithm 3 options of the timed configuration beyond the cost-model rule and depth 8:
# the 128 heaviest nodes are candidates, the side sampler takes 5 blocks per SM during
# the planning (chosen by timing the ten sources on GB300; the library defaults are 64
# and 4)
ALG3_OPTIONS = dict(alg3_max_nodes=128, alg3_overlap=5)
# Accuracy of the timed configuration as tests/test_gpu_exceed.py measured it on GB300: the same
# options (eps 1e-6, kappa 4, FP64, Algorithm 3 cost-model rule, depth <= 8) on the directed
# Chung-Lu graph of the same recipe at n = 2e4, m = 2e5 (where the Power Method gives S), 100
# seeds over five sources
ACCURACY = {"measured_by": "tests/test_gpu_exceed.py", "graph": "chung_lu n=20000 m=200000 gamma=2.1",
            "seeds": 100, "exceed_rate": 0.0, "max_err": 2.09e-7, "p50_err": 4.34e-8, "p99_err": 2.07e-7,
            "eps": 1e-6}
L2_FLUSH_BYTES = 512 << 20


def sweep_level_bytes(n, m, precision):
    """Compulsory bytes of one forward plus one reverse level."""
    csr = 4 * m + 4 * (n + 1)
    if precision == "fp64":
        return 2 * csr + (8 + 16) * n + (8 + 24) * n
    # FP32c: forward reads x (4 B), writes pi, x (8 B); reverse reads s (8 B two-float), pi (4 B),
    # w (8 B) and writes s (8 B)
    return 2 * csr + (4 + 8) * n + (8 + 4 + 8 + 8) * n


def make_graph(w):
    import synth
    if w["kind"] == "rmat":
        return synth.rmat(w["scale"], w["m"], seed=w["graph_seed"])
    if w["kind"] == "rmat_torch":
        return synth.rmat_torch(w["scale"], w["m"], seed=w["graph_seed"], device="cuda")
    if w["kind"] == "chung_lu":
        return synth.chung_lu(w["n"], w["m"], gamma=w["gamma"], seed=w["graph_seed"])
    if w["kind"] == "chung_lu_torch":
        return synth.chung_lu_torch(w["n"], w["m"], gamma=w["gamma"], seed=w["graph_seed"], device="cuda")
    return synth.erdos_renyi(w["n"], w["m"], seed=w["graph_seed"])


def sources_for(w, rp, world, rank):
    import synth
    if w["kind"] == "erdos_renyi" and w["sources"] == 1:
        return [0] * 1
    allsrc = synth.random_sources(rp, w["sources"] * world, seed=w["source_seed"])
    return [int(x) for x in allsrc[rank * w["sources"]:(rank + 1) * w["sources"]]]


def reduce_max(values, device):
    """Element-wise maximum of `values` over all ranks (identity without a process group)."""
    import torch
    import torch.distributed as dist
    t = torch.tensor(values, dtype=torch.float64, device=device)
    if dist.is_available() and dist.is_initialized() and dist.get_world_size() > 1:
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return [float(x) for x in t.cpu()]


def whole_job_rate(units_per_rank, world, max_ms):
    """Units processed by all ranks divided by the slowest rank's time (weak scaling)."""
    return units_per_rank * world / (max_ms / 1000.0)


def peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            return json.load(f), "measured"
    return {"hbm_gbs": 6800.0, "sm_max_mhz": 2070.0}, "fallback"


class ClockSampler:
    """nvidia-smi clock / throttle sampling during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device_index: int):
        self.dev = device_index
        self.proc = None
        # the raw samples go to BENCH_CLOCKS_DIR (default: the system's temporary directory);
        # the JSON line carries their summary
        out_dir = os.environ.get("BENCH_CLOCKS_DIR") or tempfile.gettempdir()
        self.path = os.path.join(out_dir, f"exactsim_clocks_rank{device_index}.csv")

    def start(self):
        try:
            os.makedirs(os.path.dirname(self.path), exist_ok=True)
            self.fh = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.dev), f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=self.fh, stderr=subprocess.DEVNULL)
        except (OSError, FileNotFoundError):
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.fh.close()
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
                for name, val in zip(names, parts[5:9]):
                    if val.lower().startswith("active"):
                        reasons.add(name)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(smax), "reasons": sorted(reasons),
                "samples": len(sm)}


def cpu_oracle_step(w, n, rp, col, u, kappa, pair_cap, threads=0):
    """One bounded sample of the CPU oracle's query for source u; returns (seconds of the
    sample, estimated seconds of the full query, info).

    The oracle runs Algorithm 1 with Algorithm 2 (its Algorithm 3 follows the paper's
    adaptive depth, whose exploration costs at least as much as the walks it replaces
    and keeps n x n supports: out of a CPU's reach at this size): forward sweeps, the
    allocation, reverse sweeps and top-k in full; the walk pairs on a sample of
    pair_cap pairs in the same per-node proportions.  Walk time is linear in the number
    of pairs, so the full query is estimated as the rest plus the sampled walk time
    times (all pairs / sampled pairs).
    """
    from oracle import linearization as lin
    from oracle import walks
    c, eps = w["c"], w["eps"]
    t0 = time.perf_counter()
    L = lin.levels(c, eps)
    H = lin.hop_vectors(n, rp, col, u, c, L)
    pi = lin.ppr(H)
    R_b = lin.sample_base(n, c, eps, kappa)
    R = lin.allocate(pi, R_b, "pi2")
    t_fwd = time.perf_counter() - t0
    total = int(R.sum())
    scale = min(1.0, pair_cap / max(total, 1))
    R_s = np.floor(R.astype(np.float64) * scale).astype(np.uint64)
    t1 = time.perf_counter()
    nonmeet, _ = walks.walk_pairs(n, rp, col, R_s, c, 1, threads)
    t_walk = time.perf_counter() - t1
    t2 = time.perf_counter()
    D = lin.dhat(nonmeet, R_s)
    s = lin.reverse(n, rp, col, H, D, c)
    lin.topk(s, w["k"], exclude=u)
    t_rev = time.perf_counter() - t2
    sampled = int(R_s.sum())
    factor = total / max(sampled, 1)
    t_step = t_fwd + t_walk + t_rev
    return t_step, t_fwd + t_rev + t_walk * factor, {"pairs_total": total, "pairs_sampled": sampled,
                                                     "walk_scale": factor, "t_sweeps_s": t_fwd + t_rev,
                                                     "t_walk_sample_s": t_walk}


def cpu_oracle_scaling_check(w, n, rp, col, u, pair_cap, threads=0):
    """A whole oracle query with no sampling (kappa small enough that all its walk pairs
    are pair_cap), against the estimate from a tenth of its pairs: the check that the
    sampled walk time scales linearly."""
    from oracle import linearization as lin
    c, eps = w["c"], w["eps"]
    L = lin.levels(c, eps)
    pi = lin.ppr(lin.hop_vectors(n, rp, col, u, c, L))
    norm_R = float(lin.allocate(pi, lin.sample_base(n, c, eps, 1.0), "pi2").sum())
    kappa = pair_cap / norm_R  # about pair_cap pairs in all
    t_full, est_full, info = cpu_oracle_step(w, n, rp, col, u, kappa, 1e30, threads)
    _, est, info_s = cpu_oracle_step(w, n, rp, col, u, kappa, info["pairs_total"] / 10.0, threads)
    return {"kappa": kappa, "pairs": info["pairs_total"], "measured_full_s": t_full,
            "estimated_from_tenth_s": est, "ratio": est / t_full}


def cpu_baseline_of(w, n, rp, col, srcs, kappa, pair_cap):
    """The oracle timed on the host cores over the workload's sources, one bounded sample
    each: (queries/s of the estimated full queries, seconds of the samples, cores, info)."""
    from oracle import walks
    walks.build()
    t_samples, t_full, infos = [], [], []
    for u in srcs:
        ts, tf, info = cpu_oracle_step(w, n, rp, col, u, kappa, pair_cap)
        t_samples.append(ts)
        t_full.append(tf)
        infos.append(info)
    return len(srcs) / sum(t_full), t_samples, walks.max_threads(), infos


def cpu_sample_note(srcs, pair_cap, infos, kappa):
    scale = statistics.mean(i["walk_scale"] for i in infos)
    return (f"oracle Algorithm 1 + Algorithm 2 at kappa={kappa:g} (the GPU path's Algorithm 3 only lowers "
            f"the variance), sources {srcs} one query each: sweeps, allocation, D^ and top-k in full, "
            f"{pair_cap:.3g} of {statistics.mean(i['pairs_total'] for i in infos):.3g} walk pairs per query on "
            f"average (same per-node proportions), walk time scaled by {scale:.3g}x to the full pair count")


def run_reference(args, w, rank, world):
    """--impl reference: the CPU oracle on the host cores (rank 0 only)."""
    if rank != 0:
        return
    from oracle import walks
    walks.build()
    n, rp, col = make_graph(w)
    srcs = sources_for(w, rp, 1, 0)
    cores = walks.max_threads()
    t_step, t_full, infos, used = [], [], [], []
    for i in range(args.warmup + args.steps):
        u = srcs[i % len(srcs)]
        ts, tf, info = cpu_oracle_step(w, n, rp, col, u, args.kappa, args.ref_pairs)
        if i >= args.warmup:
            t_step.append(ts)
            t_full.append(tf)
            infos.append(info)
            used.append(u)
    q_per_s = len(t_full) / sum(t_full)
    check = cpu_oracle_scaling_check(w, n, rp, col, srcs[0], args.ref_pairs)
    line = {
        "impl": "reference", "metric": METRIC, "value": q_per_s, "unit": "queries/s", "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1000.0 * statistics.mean(t_step),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": config_of(args, w),
        "cpu_baseline": {"value": q_per_s, "unit": "queries/s", "cores": cores, "kind": "oracle",
                         "sample": cpu_sample_note(used, args.ref_pairs, infos, args.kappa),
                         "ms_per_full_query_estimated": 1000.0 * statistics.mean(t_full),
                         "scaling_check": check},
        "e2e": {"value": q_per_s, "unit": "queries/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
        "note": "ms_per_step is the measured time of one sample step; value is 1 / the estimated time of the "
                "full query (scaling_check: a whole unsampled oracle query against its estimate)",
    }
    print(json.dumps(line), flush=True)


def sweep_roofline(esim, torch, stream, reps=5):
    """Sweep HBM GB/s on the directed Chung-Lu graph n = 4e6, m = 7e7 (gamma 2.2), FP64 and
    FP32c: forward plus reverse sweeps of one query at eps = 1e-7 (L = 33) from a seeded
    source, timed with CUDA events on the library's stream, D given (its values do not
    change the sweep's work).  The graph (0.56 GB of CSR, vectors 16-32 MB) is drawn on
    the GPU; its sweeps read more than L2 holds."""
    import synth
    wl = WORKLOADS["cl4m"]
    t0 = time.perf_counter()
    n, rp, col = synth.chung_lu_torch(wl["n"], wl["m"], gamma=wl["gamma"], seed=wl["graph_seed"], device="cuda")
    t_gen = time.perf_counter() - t0
    m = len(col)
    c = wl["c"]
    L = esim.esim_levels(c, wl["eps"])
    u = int(synth.random_sources(rp, 1, seed=wl["source_seed"])[0])
    g = esim.Graph(n, rp, col)
    g.set_stream(stream)
    del rp, col
    hist64 = torch.empty((L + 1) * n, dtype=torch.float64, device="cuda")
    hist32 = torch.empty((L + 1) * n, dtype=torch.float32, device="cuda")
    dh = torch.from_numpy(synth.uniform_diagonal(n, c, seed=3)).cuda()
    s64 = torch.empty(n, dtype=torch.float64, device="cuda")
    s32 = torch.empty(n, dtype=torch.float64, device="cuda")
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(6)]
    out = {}
    pk, pk_src = peaks()
    for prec in ("fp64", "fp32c"):
        fwd, rev = [], []
        for i in range(reps + 1):
            ev[0].record(stream)
            if prec == "fp64":
                g.forward(u, c, L, hist64)
                ev[1].record(stream)
                g.reverse(hist64, L, c, dh, s64)
            else:
                g.forward_f32(u, c, L, hist32)
                ev[1].record(stream)
                g.reverse_f32(hist32, L, c, dh, s32)
            ev[2].record(stream)
            ev[2].synchronize()
            if i > 0:  # the first pass warms up
                fwd.append(ev[0].elapsed_time(ev[1]))
                rev.append(ev[1].elapsed_time(ev[2]))
        g.sync()
        ms = statistics.mean(fwd) + statistics.mean(rev)
        gbs = L * sweep_level_bytes(n, m, prec) / (ms / 1000.0) / 1e9
        out[prec] = {"ms_forward": statistics.mean(fwd), "ms_reverse": statistics.mean(rev), "ms_query_sweeps": ms,
                     "gbs": gbs, "frac": gbs / pk["hbm_gbs"]}
    err = float((s32 - s64).abs().max().item())
    g.close()
    del hist64, hist32
    torch.cuda.empty_cache()
    return {"graph": f"chung_lu n={n} m={m} gamma={wl['gamma']} (torch generator, seed {wl['graph_seed']})",
            "L": L, "source": u, "bytes_per_level": {p: sweep_level_bytes(n, m, p) for p in ("fp64", "fp32c")},
            "peak_hbm_gbs": pk["hbm_gbs"], "peak_source": pk_src, "graph_gen_s": t_gen,
            "fp64": out["fp64"], "fp32c": out["fp32c"], "max_abs_diff_fp32c_vs_fp64": err,
            "note": "achieved = compulsory bytes of L forward + L reverse levels / CUDA-event time; "
                    "frac of the measured copy bandwidth"}


def run_precision(args, w):
    """Sweep throughput and error of the FP32c precision form against FP64, same D^."""
    import torch
    torch.cuda.set_device(0)
    import __graft_entry__
    __graft_entry__.build()
    import paper_2004_03493_gb300 as esim
    n, rp, col = make_graph(w)
    m = len(col)
    srcs = sources_for(w, rp, 1, 0)
    c, eps = w["c"], w["eps"]
    L = esim.esim_levels(c, eps)
    kappa = args.kappa
    g = esim.Graph(n, rp, col, kappa=kappa)
    # a stream of our own: the library's launches and the CUDA events must share one
    # (torch's legacy default stream would not order the library's work)
    stream = torch.cuda.Stream()
    g.set_stream(stream)
    hist64 = torch.empty((L + 1) * n, dtype=torch.float64, device="cuda")
    hist32 = torch.empty((L + 1) * n, dtype=torch.float32, device="cuda")
    pi = torch.empty(n, dtype=torch.float64, device="cuda")
    R = torch.zeros(n, dtype=torch.uint64, device="cuda")
    off = torch.zeros(n + 1, dtype=torch.uint64, device="cuda")
    nm = torch.zeros(n, dtype=torch.uint64, device="cuda")
    dh = torch.empty(n, dtype=torch.float64, device="cuda")
    s64 = torch.empty(n, dtype=torch.float64, device="cuda")
    s32 = torch.empty(n, dtype=torch.float64, device="cuda")
    R_b = esim.esim_sample_base(n, c, eps, kappa)
    per_source = []
    t = {"fp64": [], "fp32c": []}

    def timed(fn):
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        fn()
        e1.record(stream)
        e1.synchronize()
        return e0.elapsed_time(e1)

    for u in srcs:
        # D^ sampled once (FP64 forward + allocation + walks) and shared by both forms
        g.forward(u, c, L, hist64)
        g.allocate(hist64, L, R_b, 0, pi, R, off)
        g.sample(off, c, 1, nm)
        g.dhat(nm, off, dh)
        g.sync()
        pairs = int(off[n].item())
        for rep in range(args.warmup + args.steps):
            a = timed(lambda: (g.forward(u, c, L, hist64), g.reverse(hist64, L, c, dh, s64)))
            b = timed(lambda: (g.forward_f32(u, c, L, hist32), g.reverse_f32(hist32, L, c, dh, s32)))
            if rep >= args.warmup:
                t["fp64"].append(a)
                t["fp32c"].append(b)
        g.sync()
        err = float((s32 - s64).abs().max().item())
        per_source.append({"u": u, "max_abs_err_fp32c_vs_fp64": err, "pairs_for_dhat": pairs,
                           "s_u": float(s64[u].item())})
    out = {}
    pk, pk_src = peaks()
    for prec in ("fp64", "fp32c"):
        ms = statistics.mean(t[prec])
        gbs = L * sweep_level_bytes(n, m, prec) / (ms / 1000.0) / 1e9
        out[prec] = {"ms_per_query_sweeps": ms, "sweep_gbs": gbs, "frac_of_hbm": gbs / pk["hbm_gbs"]}
    line = {"metric": "sweep HBM GB/s, FP32c vs FP64 (same sources, same D^)", "value": out["fp32c"]["sweep_gbs"],
            "unit": "GB/s", "n_gpus": 1, "steps": args.steps, "warmup": args.warmup, "higher_is_better": True,
            "dtype": "f32+two-float", "data": "synthetic",
            "config": {"workload": "cl4m", "graph": "chung_lu", "n": n, "m": m, "gamma": w["gamma"], "c": c,
                       "eps": eps, "L": L, "kappa_for_dhat": kappa, "sources": srcs,
                       "l2": "inputs larger than L2 (in- and out-CSR 0.56 GB)"},
            "forms": out, "per_source": per_source,
            "error_bound_fp32c": 2.0 ** -24 * (2 * c / (1 - c) ** 2 + 2 / (1 - c)),
            "peak_hbm_gbs": pk["hbm_gbs"], "peak_source": pk_src}
    print(json.dumps(line), flush=True)
    g.close()


def run_batched(args, w):
    """Batched FP32c queries (64 per launch) against plain FP64 single queries, same sources, eps, seed, kappa."""
    import torch
    torch.cuda.set_device(0)
    import __graft_entry__
    __graft_entry__.build()
    import paper_2004_03493_gb300 as esim
    n, rp, col = make_graph(w)
    rng = np.random.default_rng(w["source_seed"] + 1)
    srcs = sources_for(w, rp, 1, 0)
    eps = np.exp(rng.uniform(np.log(w["eps_lo"]), np.log(w["eps_hi"]), size=len(srcs)))
    c, k = w["c"], w["k"]
    gb = esim.Graph(n, rp, col, kappa=args.kappa, timing=1)
    gs = esim.Graph(n, rp, col, kappa=args.kappa, timing=1)
    stream = torch.cuda.Stream()  # shared by the library's launches and the CUDA events
    gb.set_stream(stream)
    gs.set_stream(stream)
    B = len(srcs)
    ids = torch.empty(B * k, dtype=torch.int32, device="cuda")
    vals = torch.empty(B * k, dtype=torch.float64, device="cuda")
    ids1 = torch.empty(k, dtype=torch.int32, device="cuda")
    vals1 = torch.empty(k, dtype=torch.float64, device="cuda")
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device="cuda")

    def timed(fn):
        flush.zero_()
        torch.cuda.synchronize()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        fn()
        e1.record(stream)
        e1.synchronize()
        return e0.elapsed_time(e1)

    def batch():
        gb.topk_batch_device(srcs, eps, c, k, 1, ids, vals)

    def singles():
        for q in range(B):
            gs.topk_device(srcs[q], c, float(eps[q]), k, 1, ids1, vals1)

    tb, ts, bstats = [], [], []
    for i in range(args.warmup + args.steps):
        a = timed(batch)
        st = gb.stats()
        b = timed(singles)
        if i >= args.warmup:
            tb.append(a)
            ts.append(b)
            bstats.append(st)
    # walks shared across the columns (the default) against each column sampling its own
    gb.set_option("shared_walks", 0)
    t_unshared = timed(batch)
    st_unshared = gb.stats()
    gb.set_option("shared_walks", 1)
    # accuracy of the batched form against the plain FP64 single queries on the same walks
    sb = gb.query_batch(srcs[:8], eps[:8], c, seed=1)
    diffs = [float(np.max(np.abs(sb[q] - gs.query(srcs[q], c, float(eps[q]), 1)))) for q in range(8)]
    qb = B / (statistics.mean(tb) / 1000.0)
    qs = B / (statistics.mean(ts) / 1000.0)
    # sweep roofline of the batched form: compulsory bytes of the n x W forward and reverse levels
    # (CSR once per level, FP32 X read and hist/X written forward; two-float s read and written,
    # FP32 hist and two-float w read reverse) over the batch's forward and reverse phases
    Wd = 64 if B > 32 else (32 if B > 16 else 16)
    Lmax = max(esim.esim_levels(c, float(e)) for e in eps)
    csr = 4 * len(col) + 4 * (n + 1)
    bytes_fwd = csr + (4 + 8) * n * Wd
    bytes_rev = csr + (8 + 4 + 8 + 8) * n * Wd
    ms_f = statistics.mean(s_["ms_forward"] for s_ in bstats)
    ms_r = statistics.mean(s_["ms_reverse"] for s_ in bstats)
    pk, pk_src = peaks()
    gbs_b = Lmax * (bytes_fwd + bytes_rev) / ((ms_f + ms_r) / 1000.0) / 1e9
    line = {"metric": "top-k queries/s, batched FP32c (64 per launch) vs plain FP64 single queries", "value": qb,
            "unit": "queries/s", "n_gpus": 1, "steps": args.steps, "warmup": args.warmup, "higher_is_better": True,
            "dtype": "f32+two-float", "data": "synthetic",
            "config": {"workload": "rmat20", "graph": "rmat", "n": n, "m": len(col), "abcd": [0.57, 0.19, 0.19, 0.05],
                       "c": c, "eps": f"log-uniform [{w['eps_lo']:g}, {w['eps_hi']:g}]",
                       "eps_config": f"log-uniform [{w['eps_config'][0]:g}, {w['eps_config'][1]:g}]",
                       "eps_note": "kappa 4 (the exceed-rate test's setting) without Algorithm 3 in the batch "
                                   "path affords eps >= 1e-5: at 1e-7 the source alone needs about 2.8e14 pairs",
                       "sources_per_launch": B, "top_k": k,
                       "kappa": args.kappa, "l2": "flushed (512 MB write) before each timed step",
                       "batch_tile_fwd": gb.get_option("batch_tile_fwd64"),
                       "batch_tile_rev": gb.get_option("batch_tile_rev64")},
            "batched_fp32c_qps": qb, "single_fp64_qps": qs, "speedup": qb / qs,
            "sweep_roofline": {"bound": "hbm", "achieved": gbs_b, "peak": pk["hbm_gbs"], "unit": "GB/s",
                               "frac": gbs_b / pk["hbm_gbs"], "peak_source": pk_src, "L_max": Lmax, "W": Wd,
                               "note": "compulsory bytes of the L_max forward and reverse n x W levels over the "
                                       "batch's forward and reverse phases (CUDA events)"},
            "batched_phases_ms": {p: statistics.mean(s_[f"ms_{p}"] for s_ in bstats)
                                  for p in ("forward", "allocate", "sample", "reverse", "topk")},
            "max_abs_diff_batched_vs_single_first8": max(diffs),
            "shared_walks": {"pairs": statistics.mean(s_["sum_R"] for s_ in bstats),
                             "pairs_unshared": st_unshared["sum_R"],
                             "sample_ms": statistics.mean(s_["ms_sample"] for s_ in bstats),
                             "sample_ms_unshared": st_unshared["ms_sample"], "ms_unshared": t_unshared,
                             "note": "same per-column counts either way (the walk spec keys pairs by node and "
                                     "index); shared: one walk set per node cut at the distinct R_q(k)"},
            "note": "both forms draw the same walk pairs (one seed); the difference is FP32c rounding plus "
                    "the sampling noise of R(k) decided from FP32 pi"}
    print(json.dumps(line), flush=True)
    gb.close()
    gs.close()


def run_serving(args, w):
    """Continuous-batching server under Poisson arrivals: p50/p99 latency and queries/s per rate."""
    import threading
    import torch
    torch.cuda.set_device(0)
    import __graft_entry__
    __graft_entry__.build()
    import paper_2004_03493_gb300 as esim
    t_gen = time.perf_counter()
    n, rp, col = make_graph(w)
    torch.cuda.empty_cache()
    t_gen = time.perf_counter() - t_gen
    t_load = time.perf_counter()
    g = esim.Graph(n, rp, col)
    t_load = time.perf_counter() - t_load
    m = len(col)
    srcs = synth_sources(rp, w["sources"], w["source_seed"])
    del rp, col
    c, k = w["c"], w["k"]
    rng = np.random.default_rng(11)
    srv = esim.Server(g, c, k=k, seed=1, kappa=args.kappa, max_batch=args.max_batch, max_waves=args.max_waves)
    # warm-up: one wave per width the run will use (tunes the batched tiles)
    for u in srcs[:args.max_batch]:
        srv.submit(int(u), 1e-5)
    ids = np.empty(k, dtype=np.int32)
    vals = np.empty(k, dtype=np.float64)
    results = []
    rates = [float(x) for x in args.rates.split(",")]
    per_rate = []
    while True:
        st0 = srv.stats()
        if st0["completed"] + st0["failed"] >= args.max_batch:
            break
        time.sleep(0.05)
    base = srv.stats()
    si = args.max_batch
    for lam in rates:
        rids = []
        t0 = time.perf_counter()
        nxt = t0
        while nxt - t0 < args.duration:
            now = time.perf_counter()
            if nxt > now:
                time.sleep(nxt - now)
            u = int(srcs[si % len(srcs)])
            si += 1
            e = float(rng.choice(w["eps_set"]))
            rids.append(srv.submit(u, e))
            nxt += rng.exponential(1.0 / lam)
        lat = []
        for r in rids:
            lat.append(srv.wait(r, 600000)[2])
        t_end = time.perf_counter()
        st = srv.stats()
        lat = np.array(lat)
        per_rate.append({"rate_qps": lam, "submitted": len(rids), "queries_per_s": len(rids) / (t_end - t0),
                         "p50_ms": float(np.percentile(lat, 50)), "p99_ms": float(np.percentile(lat, 99)),
                         "max_ms": float(lat.max()), "waves": st["waves"] - base["waves"],
                         "mean_batch": st["mean_batch"], "max_running": st["max_running"]})
        base = st
    srv.close()
    best = max(per_rate, key=lambda r: r["queries_per_s"])
    line = {"metric": "served top-100 queries/s with p50/p99 latency (Poisson arrivals)", "value": best["queries_per_s"],
            "unit": "queries/s", "n_gpus": 1, "higher_is_better": True, "dtype": "f32+two-float", "data": "synthetic",
            "config": {"workload": "rmat25", "graph": "rmat (torch generator)", "n": n, "m": m,
                       "abcd": [0.57, 0.19, 0.19, 0.05], "c": c, "eps": list(w["eps_set"]),
                       "eps_config": list(w["eps_config"]),
                       "eps_note": "kappa 4 (the exceed-rate test's setting) without Algorithm 3 in the batch path: "
                                   "a request at eps 1e-6 needs about 3.5e12 walk pairs on this graph",
                       "top_k": k,
                       "kappa": args.kappa, "max_batch": args.max_batch, "max_waves": args.max_waves,
                       "duration_s_per_rate": args.duration},
            "rates": per_rate, "graph_gen_s": t_gen, "graph_load_s": t_load}
    print(json.dumps(line), flush=True)
    g.close()


def synth_sources(rp, count, seed):
    import synth
    return synth.random_sources(rp, count, seed=seed)


def config_of(args, w):
    return {"workload": args.workload, "graph": w["kind"], "n": w["n"], "m": w["m"],
            "gamma": w.get("gamma"), "c": w["c"], "eps": w["eps"], "sources": w["sources"], "queries_per_step": 1,
            "top_k": w["k"], "kappa": args.kappa, "alloc": "pi^2 (Lemma 4)",
            "dhat": (f"Algorithm 3, the library's cost-model rule (alg3_rule 1): exact Z_1..Z_d for the "
                     f"{ALG3_OPTIONS['alg3_max_nodes']} heaviest nodes at a cost-chosen d <= 8, "
                     "max(1, ceil(R_b pi^2 c^(2d))) tail walk pairs; the others Algorithm 2"
                     if getattr(args, "alg3", 0) else "Algorithm 2 (walk pairs)"),
            "alg3_options": ALG3_OPTIONS if getattr(args, "alg3", 0) else None,
            "accuracy": ACCURACY,
            "l2": "flushed (512 MB write) before each timed step", "parallelism": f"replicas x{args.gpus}"}


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="cl100k", choices=sorted(WORKLOADS))
    ap.add_argument("--kappa", type=float, default=4.0,
                    help="sample constant: R_b = kappa ln(n) / eps^2 (<= 0: the paper's 6/(1-sqrt c)^4)")
    ap.add_argument("--ref-pairs", type=float, default=5e7, help="walk pairs per CPU oracle sample")
    ap.add_argument("--no-sweeps", action="store_true", help="leave out the n=4e6 sweep roofline")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--precision", type=int, default=0, help="0: FP64 sweeps; 1: FP32c")
    ap.add_argument("--alg3", type=int, default=1,
                    help="1 (default): Algorithm 3 D^ estimator for the heaviest nodes; 0: Algorithm 2 only")
    ap.add_argument("--rates", default="1,4", help="serving: Poisson arrival rates (queries/s), comma-separated")
    ap.add_argument("--duration", type=float, default=20.0, help="serving: seconds of arrivals per rate")
    ap.add_argument("--max-batch", type=int, default=8, help="serving: requests per wave")
    ap.add_argument("--max-waves", type=int, default=2, help="serving: waves in flight")
    args = ap.parse_args()
    w = WORKLOADS[args.workload]

    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))

    if args.impl == "reference":
        run_reference(args, w, rank, world)
        return
    if args.workload == "cl4m":
        run_precision(args, w)
        return
    if args.workload == "rmat20":
        run_batched(args, w)
        return
    if args.workload == "rmat25":
        run_serving(args, w)
        return

    import torch
    import torch.distributed as dist
    if world > 1:
        torch.cuda.set_device(local_rank)
        dist.init_process_group("nccl", device_id=torch.device("cuda", local_rank))
    else:
        torch.cuda.set_device(0)
    dev = torch.device("cuda", torch.cuda.current_device())

    import __graft_entry__
    if rank == 0:
        __graft_entry__.build()
    if world > 1:
        dist.barrier()
    if rank != 0:
        __graft_entry__.build()
    import paper_2004_03493_gb300 as esim

    n, rp, col = make_graph(w)
    srcs = sources_for(w, rp, world, rank)
    c, eps, k = w["c"], w["eps"], w["k"]
    g = esim.Graph(n, rp, col, kappa=args.kappa, timing=1, alg3=args.alg3, alg3_rule=1, alg3_max_depth=8,
                   **ALG3_OPTIONS)
    stream = torch.cuda.Stream(device=dev)  # shared by the library's launches and the CUDA events
    g.set_stream(stream)
    ids = torch.empty(k, dtype=torch.int32, device=dev)
    vals = torch.empty(k, dtype=torch.float64, device=dev)
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device=dev)

    # One step = one top-k query through the public host API (host output buffers; the
    # query parameters pass by value, the k ids and scores come back every step).  The
    # sources cycle through the workload's list; CUDA events on the library's stream
    # time the device work, the host clock times the whole call (end to end).
    host_ids = np.empty(k, dtype=np.int32)
    host_vals = np.empty(k, dtype=np.float64)

    def step(i):
        u = srcs[i % len(srcs)]
        esim.esim_topk(g.handle, u, c, eps, i, k, host_ids, host_vals)

    # the clock sampler starts before the warm-up so that nvidia-smi's start-up cost stays
    # out of the timed region
    clocks = ClockSampler(torch.cuda.current_device())
    clocks.start()
    for i in range(args.warmup):
        step(i)
    torch.cuda.synchronize()
    stats = []
    step_ms = []
    e2e_s = 0.0
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    t_wall0 = time.perf_counter()
    for i in range(args.steps):
        flush.zero_()
        ev0 = torch.cuda.Event(enable_timing=True)
        ev1 = torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        ev0.record(stream)
        step(args.warmup + i)
        ev1.record(stream)
        ev1.synchronize()
        e2e_s += time.perf_counter() - t0
        step_ms.append(ev0.elapsed_time(ev1))
        stats.append(g.stats())
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    wall = time.perf_counter() - t_wall0
    clk = clocks.stop()
    total_ms = float(sum(step_ms))

    total_ms, e2e_s = reduce_max([total_ms, e2e_s], dev)
    queries = args.steps * world
    value = whole_job_rate(args.steps, world, total_ms)

    # roofline of the dominant kernel (the walk-pair sampler): pair-steps per second against
    # the rate of the Philox-4x32-10 blocks alone, one a step;
    # the sampler's launches: with Algorithm 3 one on the side stream (the walks whose plan is
    # final, overlapping the planning) and one after the planning; achieved = pair-steps /
    # the sum of the launches' durations (CUDA events on each launch's own stream)
    steps_total = sum(s["pair_steps"] for s in stats)
    ms_sample = sum(s["ms_sample_kernel"] + s["ms_sample_side"] for s in stats)
    sampler_launches = sum(1 + (1 if s["pair_steps_side"] else 0) for s in stats)
    ms_phase = {p: sum(s[f"ms_{p}"] for s in stats) for p in ("forward", "allocate", "sample", "reverse", "topk")}
    pk, pk_src = peaks()
    sm_max = float(pk.get("sm_max_mhz", 2070.0))
    sm_count = torch.cuda.get_device_properties(dev).multi_processor_count
    peak_steps = sm_count * sm_max * 1e6 * PHILOX_PER_SM_CLOCK
    achieved = steps_total / (ms_sample / 1000.0) if ms_sample > 0 else 0.0
    L = stats[0]["L"] if stats else 0
    # compulsory bytes of one forward plus one reverse FP64 level: each reads its CSR
    # (4 B per entry, 4 B per row pointer) and its input vector once (8 B per node); the
    # forward level writes pi^l and x^l (16 B per node), the reverse level reads pi^(L-l)
    # and D^ and writes s^l (24 B per node)
    m_edges = len(col)
    sweep_bytes = sweep_level_bytes(n, m_edges, "fp64")
    sweep_gbs = (len(stats) * L * sweep_bytes) / ((ms_phase["forward"] + ms_phase["reverse"]) / 1000.0) / 1e9 \
        if stats else 0.0
    launches = sum(s["launches"] for s in stats)
    # Lemma 2 with the pi^2 allocation: Var s(v) <= ||pi_v||^2 / (4 a^4 R_b) (using D(1-D) <= 1/4);
    # ||pi_v||^2 <= 1 bounds every node, ||pi_u||^2 (measured) the source itself
    a = 1.0 - math.sqrt(c)
    R_b = stats[0]["R_b"] if stats else 0.0
    norm_u = statistics.mean(s["pi_norm2"] for s in stats) if stats else 0.0
    sigma_u = math.sqrt(norm_u / (4 * a ** 4 * R_b)) if R_b > 0 else None
    sigma_any = math.sqrt(1.0 / (4 * a ** 4 * R_b)) if R_b > 0 else None
    line = {
        "metric": METRIC, "value": value, "unit": "queries/s", "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": total_ms / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic", "config": config_of(args, w),
        "clocks": clk,
        "e2e": {"value": queries / e2e_s, "unit": "queries/s", "h2d_bytes_per_step": 0,
                "d2h_bytes_per_step": k * (4 + 8),
                "note": "host clock around esim_topk with host output buffers; query parameters pass by value"},
        "gpu_launches": launches,
        "roofline": {"kernel": "sample_pairs_kernel", "launches": sampler_launches,
                     "ms_per_launch": ms_sample / max(sampler_launches, 1),
                     "bound": "alu", "achieved": achieved / 1e9,
                     "peak": peak_steps / 1e9, "unit": "G pair-steps/s", "frac": achieved / peak_steps,
                     "traffic": SAMPLER_TRAFFIC,
                     "peak_source": f"{sm_count} SMs x {sm_max:.0f} MHz ({pk_src} clock) x {PHILOX_PER_SM_CLOCK:.3f} "
                                    "Philox-4x32-10 blocks per SM and clock, as a kernel that only draws them runs"},
        "phases_ms": {p: v / max(len(stats), 1) for p, v in ms_phase.items()},
        "walk": {"pairs_per_query": sum(s["sum_R"] for s in stats) / max(len(stats), 1),
                 "pair_steps_per_s": achieved, "L": L, "R_b": R_b},
        "error_bound": {"sigma_source": sigma_u, "sigma_any_node": sigma_any, "eps": eps,
                        "note": "Lemma 2 variance bound with the pi^2 allocation at this kappa; "
                                "kappa = 6/(1-sqrt c)^4 carries Theorem 1's guarantee"},
        "sweep_hbm_gbs_cl100k": sweep_gbs,
        "wall_s": wall,
    }
    if rank == 0 and world == 1 and not args.no_sweeps:
        line["sweep_roofline"] = sweep_roofline(esim, torch, stream)
        line["sweep_hbm_gbs_fp64"] = line["sweep_roofline"]["fp64"]["gbs"]
        line["sweep_hbm_gbs_fp32c"] = line["sweep_roofline"]["fp32c"]["gbs"]
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        qps, t_samples, cores, infos = cpu_baseline_of(w, n, rp, col, srcs, args.kappa, args.ref_pairs)
        line["cpu_baseline"] = {"value": qps, "unit": "queries/s", "cores": cores, "kind": "oracle",
                                "sample": cpu_sample_note(srcs, args.ref_pairs, infos, args.kappa),
                                "sample_s": sum(t_samples)}
    if rank == 0:
        print(json.dumps(line), flush=True)
    g.close()
    if world > 1:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
