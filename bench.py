#!/usr/bin/env python3
"""Benchmark: all-edge spanning centrality (AESC) edges/s on one GB300.

Workload (default): Barabasi-Albert graph, n = 200,000, 10 edges per new node
(m = 1,999,900), seed 1; FP32 probability blocks with FP64 edge accumulation;
eps = 1e-3; per-source lengths from the MLP (trained beforehand on another
Barabasi-Albert graph, n = 50,000, seed 101), every edge certified by the
a-posteriori bound and extended when it fails, capped by the length of Eq. (6).

A step is one full sc_all_edges call: every edge's s_hat, all sources. The
eigenvalue bound, the features and the model are preprocessing (computed once
per graph or graph family, outside the timed region, as the paper separates
preprocessing from the run). The plain global-length arms (FP32 and FP64) are
timed beside it for comparison.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]
    python bench.py --mode tgt_plus --policy global     # Algorithm 4 on the same workload

Prints one JSON line on rank 0. With N > 1 (torchrun) every rank runs an
independent replica on its own GPU (the method has no exchange step between
sources: replicas only), value = all ranks' edges / max rank time.
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
sys.path.insert(0, ROOT)

METRIC = "AESC edges/sec at \u03b5=1e-3 (learned-\u2113 FP32 batched vs plain global-\u2113); HBM GB/s"
UNIT = "edges/s"
WORKLOADS = {
    "ba_200k": dict(desc="Barabasi-Albert n=200000, 10 edges per new node (m=1,999,900), seed 1",
                    make=lambda gg: gg.barabasi_albert(200_000, 10, 1)),
    "tree_gnp_2k": dict(desc="uniform random tree + G(n,p), n=2000, avg degree 10, seed 0",
                        make=lambda gg: gg.tree_plus_gnp(2000, 10.0, 0)),
    "lattice_1000": dict(desc="1000x1000 lattice, 5% of edges deleted outside a random spanning tree, seed 2 "
                              "(bipartite, bandwidth 1000)",
                         make=lambda gg: gg.perturbed_grid(1000, 1000, 0.05, 2)),
    "rmat_22": dict(desc="R-MAT scale 22, (a,b,c,d) = (.57,.19,.19,.05), edge factor 16, symmetrised, largest "
                         "component (n = 2,394,610, m = 64,153,249), seed 5",
                    make=lambda gg: gg.rmat(22)),
}
# the graph each workload's learned-length model is trained on (same family, another seed)
TRAIN_GRAPHS = {
    "rmat_22": ("R-MAT scale 16 seed 15", lambda gg: gg.rmat(16, seed=15)),
    "lattice_1000": ("200x200 lattice, 5% of edges deleted, seed 102 (labels from the tail estimate, cap 511)",
                     lambda gg: gg.perturbed_grid(200, 200, 0.05, 102)),
}
TRAIN_CAP = 511  # label cap of a bipartite training graph (sc_estimated_lengths)
# the batch's model: one graph of each family of the batch (other seeds); the lattice's labels
# at eps = 1e-3 reach a few thousand hops, hence the larger cap
BATCH_TRAIN = ("G(n, 8/(n-1)) LCC n=5000 seed 901, Barabasi-Albert n=5000 m=5 seed 902, 70x70 lattice seed 903 "
               "(labels from the tail estimate, cap 4095)",
               lambda gg: [gg.gnp_lcc(5000, 8.0, 901), gg.barabasi_albert(5000, 5, 902),
                           gg.perturbed_grid(70, 70, 0.05, 903)])
BATCH_TRAIN_CAP = 4095
DEFAULT_TRAIN = ("Barabasi-Albert n=50000 m0=10 seed 101", lambda gg: gg.barabasi_albert(50_000, 10, 101))
KERNEL_SOURCES = ["paper_2305_16086_gb300/csrc/propagate.cuh", "paper_2305_16086_gb300/csrc/hop2_mask.cuh",
                  "paper_2305_16086_gb300/csrc/sparse_hops.cuh"]
# kernel classes the library times separately (SC_KC_* order) and their kernels
KERNEL_CLASSES = {"dense_hop": "k_spmm_hop", "mask_hop": "k_front_scatter + k_front2, or k_mask_scatter + k_hop2_mask", "sparse_hop": "k_front3",
                  "ball_hop": "k_ball_rows + k_ball", "last_hop": "k_last_hop",
                  "switch_test": "k_chi_tiles + k_chi_column + k_chi_entries "
                                 "(+ the sums' copy and the host's wait)",
                  "walks": "k_walk_plan + k_walk_chunks + k_walk_finish"}
TRAFFIC_FILE = os.path.join(ROOT, "profiles", "spmm_hop_ba200k_traffic.json")


def kernel_source_sha() -> str:
    """Hash of the hop kernel's code with comments and blank space removed
    (a comment edit does not make recorded counters stale)."""
    import re

    h = hashlib.sha256()
    for rel in KERNEL_SOURCES:
        with open(os.path.join(ROOT, rel), encoding="utf-8") as fh:
            text = fh.read()
        text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
        text = re.sub(r"//[^\n]*", "", text)
        h.update("\n".join(l.strip() for l in text.splitlines() if l.strip()).encode())
    return h.hexdigest()[:16]


def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as fh:
            d = json.load(fh)
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


def recorded_traffic(config_key: str):
    """DRAM bytes per launch from the committed ncu summary, if it was taken
    on the current kernel source and the same launch configuration."""
    try:
        with open(TRAFFIC_FILE) as fh:
            d = json.load(fh)
    except Exception:
        return None
    if d.get("kernel_source_sha") != kernel_source_sha():
        return None
    return d.get("configs", {}).get(config_key)


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device_index: int):
        self.dev = device_index
        self.proc = None
        self.path = os.path.join(tempfile.gettempdir(), f"sc_bench_clocks_{os.getpid()}.csv")

    def __enter__(self):
        try:
            os.makedirs(os.path.dirname(self.path), exist_ok=True)
            self.fh = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                                          "-i", str(self.dev), "-lms", "200"], stdout=self.fh,
                                         stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None
        return self

    def __exit__(self, *exc):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()
            self.fh.close()

    def summary(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        rows = []
        with open(self.path) as fh:
            for line in fh:
                parts = [p.strip() for p in line.split(",")]
                if len(parts) >= 9:
                    rows.append(parts)
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        smax = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if r[5 + i].lower() == "active"})
        loaded = [v for v in sm if smax and v > 0.5 * max(smax)] or sm
        return {"sm_mhz": statistics.median(loaded) if loaded else None,
                "sm_max_mhz": max(smax) if smax else None, "reasons": reasons, "samples": len(rows)}


def cpu_baseline(g, ell: int, target_s: float = 10.0):
    """The oracle's Algorithm 2 (oracle.series.half_sums, FP64, OpenMP over
    sources) timed on a bounded sample of sources at the bench's length."""
    from oracle import _native, series

    threads = _native.default_threads()
    rng = np.random.default_rng(123)
    sample = max(threads, 16)
    elapsed = 0.0
    done = 0
    while True:
        src = rng.choice(g.n, size=min(sample, g.n), replace=False)
        t0 = time.perf_counter()
        series.half_sums(g.n, g.row_ptr, g.col_idx, ell, sources=src, extra_steps=0, threads=threads)
        dt = time.perf_counter() - t0
        elapsed += dt
        done += src.size
        if elapsed >= target_s or src.size >= g.n:
            break
        sample = int(min(g.n, max(src.size * 2, src.size * (target_s - elapsed) / max(dt, 1e-3))))
    per_source = elapsed / done
    value = g.m / (per_source * g.n)
    return {"value": value, "unit": UNIT, "cores": threads, "kind": "oracle",
            "sample": f"{done} sources drawn from {g.n} (Algorithm 2 in FP64 C, length {ell}); "
                      f"full-job rate = m / (n * seconds per source)", "seconds": round(elapsed, 2),
            "sources_timed": done}


def exact_check(g, s_hat, edges: int, seed: int = 2024):
    """The exact resistance (oracle O1: Jacobi-preconditioned FP64 CG on the
    Laplacian, one solve per edge) on `edges` uniformly sampled edges, timed on
    the host cores, and the error of the GPU result s_hat (one value per CSR
    entry) there: max and mean |s_hat - r|. Part of the CPU baseline leg."""
    from oracle import _native, exact

    e = g.edges()
    rng = np.random.default_rng(seed)
    pick = e[rng.choice(e.shape[0], size=min(edges, e.shape[0]), replace=False)]
    k = exact.entry_of_edges(g.n, g.row_ptr, g.col_idx, pick)
    t0 = time.perf_counter()
    r = exact.exact_cg(g.n, g.row_ptr, g.col_idx, pick)
    dt = time.perf_counter() - t0
    err = np.abs(np.asarray(s_hat)[k] - r)
    return {"sampled_edges": int(pick.shape[0]), "max_abs_err": float(err.max()), "mean_abs_err": float(err.mean()),
            "oracle": "FP64 Jacobi-preconditioned CG per sampled edge, relative residual 1e-12",
            "oracle_seconds": round(dt, 2), "oracle_edges_per_s": pick.shape[0] / dt,
            "oracle_cores": _native.default_threads(), "sample_seed": seed}


def train_model(eps, stream, workload="ba_200k"):
    """The MLP for the learned length, trained on the GPU on a separate graph of
    the same family (untimed preprocessing)."""
    import graphgen as gg
    from paper_2305_16086_gb300 import Graph, binding

    tg = TRAIN_GRAPHS.get(workload, DEFAULT_TRAIN)[1](gg)
    bip = bool(tg.meta.get("bipartite"))
    with Graph(tg.row_ptr, tg.col_idx, stream=stream) as Gt:
        Gt.estimate_lambda(allow_unconverged=bip)  # a bipartite graph's labels do not use lambda
        init = np.random.default_rng(0).normal(0.0, 0.2, binding.MLP_PARAMS).astype(np.float32)
        model, _ = binding.mlp_train([Gt], init, epochs=400, lr=1e-2, eps=eps, precision="fp32",
                                     ell_cap=TRAIN_CAP if bip else 0)
    return model


def lattice_reference(g, edges: int, seed: int = 2024):
    """Exact resistances (oracle O1, sparse LU of the grounded Laplacian, one
    process per host core) on `edges` uniformly sampled edges of a lattice,
    where CG converges slowly. Part of the CPU baseline leg."""
    from oracle import _native, exact

    e = g.edges()
    rng = np.random.default_rng(seed)
    pick = e[rng.choice(e.shape[0], size=min(edges, e.shape[0]), replace=False)]
    k = exact.entry_of_edges(g.n, g.row_ptr, g.col_idx, pick)
    t0 = time.perf_counter()
    r = exact.exact_sparse_lu(g.n, g.row_ptr, g.col_idx, pick, processes=_native.default_threads())
    return {"pick": pick, "k": k, "r": r, "seconds": time.perf_counter() - t0, "seed": seed,
            "cores": _native.default_threads()}


def errors_at(ref, s_hat):
    err = np.abs(np.asarray(s_hat)[ref["k"]] - ref["r"])
    return {"sampled_edges": int(ref["k"].size), "max_abs_err": float(err.max()), "mean_abs_err": float(err.mean())}


def empirical_length(G, ref, eps, cap, kw):
    """The global judge on a slow-mixing graph: the least odd length whose
    end-corrected series is within eps of the exact values on the sampled
    edges (bisection: the end-corrected series grows with the length), from the
    GPU series at the sampled entries (sc_some_edges)."""
    from paper_2305_16086_gb300 import binding

    def ok(ell):
        s, _ = binding.some_edges(G, ref["k"], **dict(kw, policy="fixed", ell_fixed=ell))
        return np.max(np.abs(s - ref["r"])) <= eps

    lo, hi = 0, (cap - 1) // 2  # odd lengths 2 i + 1, i in [lo, hi]
    if not ok(2 * hi + 1):
        return None
    while lo < hi:
        mid = (lo + hi) // 2
        if ok(2 * mid + 1):
            hi = mid
        else:
            lo = mid + 1
    return 2 * lo + 1


def dist_setup():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def max_over_ranks(pg, x: float, device) -> float:
    """The slowest rank's value (the job ends when the last replica does)."""
    if pg is None:
        return x
    import torch

    t = torch.tensor([x], device=device, dtype=torch.float64)
    pg.all_reduce(t, op=pg.ReduceOp.MAX)
    return float(t.item())


def replica_value(world: int, m: int, ms_per_step: float) -> float:
    """Whole-job edges/s: every replica processes all m edges of its own copy
    of the workload per step (weak scaling, no exchange between replicas)."""
    return world * m / (ms_per_step / 1e3)


def timed_passes(run_pass, warm: int, timed: int, sync, barrier):
    """Run `warm` + `timed` passes of run_pass(mark); run_pass calls mark(name)
    after each of its phases. The warm-up passes synchronize at every mark and
    return the last one's phase times (ms); the timed passes run without those
    synchronizations and return their wall times (ms), each bracketed by a
    barrier and a synchronize."""
    times, phases = [], {}
    for i in range(warm + timed):
        split = i < warm
        marks = []

        def mark(name):
            if split:
                sync()
                marks.append((name, time.perf_counter()))

        barrier()
        t0 = time.perf_counter()
        run_pass(mark)
        sync()
        if split:
            prev, phases = t0, {}
            for name, t in marks:
                phases[name] = round((t - prev) * 1e3, 3)
                prev = t
        else:
            times.append((time.perf_counter() - t0) * 1e3)
    return times, phases


def run_reference(args, world, rank):
    """The oracle on the host cores: each step a bounded sample of the workload
    (the sources Algorithm 2 runs are drawn at random; the sample is timed and
    its rate scaled to the unit, edges per second of the whole graph)."""
    if rank != 0:
        return
    import graphgen as gg
    from oracle import truncation

    g = WORKLOADS[args.workload]["make"](gg)
    lp, lm, ls = truncation.spectrum_extremes(g.n, g.row_ptr, g.col_idx)
    ell = int(truncation.tau_entries(g.n, g.row_ptr, g.col_idx, args.eps, ls).max())
    vals = []
    for i in range(args.warmup + args.steps):
        r = cpu_baseline(g, ell, target_s=args.ref_step_seconds)
        if i >= args.warmup:
            vals.append(r)
    value = statistics.mean(v["value"] for v in vals)
    ms = 1e3 * statistics.mean(v["seconds"] for v in vals)
    sources = statistics.mean(v["sources_timed"] for v in vals)
    out = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
           "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True,
           "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
           "step": f"one step = Algorithm 2 for about {sources:.0f} randomly drawn sources of the {g.n} "
                   f"(a bounded sample); value = the sample's rate in edges of the whole graph per second",
           "full_job_ms_extrapolated": g.m / value * 1e3,
           "config": {"workload": WORKLOADS[args.workload]["desc"], "n": g.n, "m": g.m, "eps": args.eps,
                      "mode": "tgt", "policy": "global", "estimator": "plain", "windowed": False,
                      "precision": "fp64 (the oracle's Algorithm 2 in C)",
                      "batching": "OpenMP over sources", "ell_global": ell, "lambda_star": ls,
                      "parallelism": f"{vals[0]['cores']} host threads",
                      "note": "the plain global-length FP64 traversal, the comparison the metric names"},
           "cpu_baseline": {"value": value, "unit": UNIT, "cores": vals[0]["cores"], "kind": "oracle",
                            "sample": vals[0]["sample"]},
           "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(out), flush=True)


def train_batch_model(eps, stream):
    """The batch's MLP: trained on the GPU on one graph of each family of the
    batch (other seeds; untimed preprocessing)."""
    import graphgen as gg
    from paper_2305_16086_gb300 import Graph, binding

    ts = BATCH_TRAIN[1](gg)
    Gt = [Graph(t.row_ptr, t.col_idx, stream=stream) for t in ts]
    try:
        for G, t in zip(Gt, ts):
            G.estimate_lambda(allow_unconverged=bool(t.meta.get("bipartite")))
        init = np.random.default_rng(0).normal(0.0, 0.2, binding.MLP_PARAMS).astype(np.float32)
        model, _ = binding.mlp_train(Gt, init, epochs=400, lr=1e-2, eps=eps, precision="fp32",
                                     ell_cap=BATCH_TRAIN_CAP)
    finally:
        for G in Gt:
            G.close()
    return model


def batch_references(gs, workers: int):
    """Start the exact values of every graph of the batch (oracle O1: dense for
    n <= 5000, else 200 sampled edges by sparse LU for lattices or CG) in a
    spawn pool, to run on the host cores while the GPU works. Part of the CPU
    baseline leg. Returns (executor, futures)."""
    import concurrent.futures as cf
    import multiprocessing as mp

    from oracle import exact

    ex = cf.ProcessPoolExecutor(max_workers=workers, mp_context=mp.get_context("spawn"))
    futs = [ex.submit(exact.reference_values, x.n, x.row_ptr, x.col_idx, 5000, 200, 100 + i,
                      bool(x.meta.get("bipartite")), 2) for i, x in enumerate(gs)]
    return ex, futs


def run_batch(args, world, rank):
    """The many-graph workload through sc_batch_all_edges: 512 graphs, n
    log-uniform in [1e3, 5e4] (G(n, 8/(n-1)) LCC, Barabasi-Albert m = 5 and
    perturbed lattices in turn), FP32 blocks. With the learned policy (the
    default) every graph takes its lengths from one model (checked per edge:
    the bound with the graph's lambda*, on the lattices the tail estimate, cap
    --batch-cap); otherwise non-bipartite graphs take their own Eq. 6 length
    and the lattices (no Eq. 6 length) take --grid-ell. The per-graph maximum
    error against the exact values is reported (the CPU leg, computed while
    the GPU runs)."""
    import torch

    import graphgen as gg
    from paper_2305_16086_gb300 import Graph, binding

    torch.cuda.set_device(int(os.environ.get("LOCAL_RANK", "0")))
    t0 = time.perf_counter()
    gs = gg.batch_graphs(512, 1000, 50000, base_seed=4)
    gen_s = time.perf_counter() - t0
    refs_ex = refs = None
    if not args.no_cpu_baseline and rank == 0 and world == 1:
        keys = ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS")
        saved = {key: os.environ.get(key) for key in keys}
        os.environ.update({key: "2" for key in keys})  # workers of two threads share the host cores
        try:
            refs_ex, refs = batch_references(gs, max(1, (os.cpu_count() or 8) // 2 - 1))
        finally:
            for key, v in saved.items():
                if v is None:
                    os.environ.pop(key, None)
                else:
                    os.environ[key] = v
    stream = torch.cuda.current_stream()
    learned = args.policy == "learned"
    model = train_batch_model(args.eps, stream) if learned else None
    Gs = [Graph(g.row_ptr, g.col_idx, stream=stream) for g in gs]
    if learned:
        ells = None
        for G, g in zip(Gs, gs):
            G.estimate_lambda(allow_unconverged=True)
            binding.mlp_load(G, model)
    else:
        ells = [args.grid_ell if g.meta.get("bipartite") else 0 for g in gs]
        for G, e in zip(Gs, ells):
            if e == 0:
                G.estimate_lambda(allow_unconverged=True)
    kw = dict(eps=args.eps, precision=args.precision, estimator="end_corrected",
              policy="learned" if learned else "global", ell_cap=args.batch_cap)
    for _ in range(args.warmup):
        binding.batch_all_edges(Gs, ells, **kw)
    torch.cuda.synchronize()
    times, reps, outs = [], None, None
    with ClockSampler(torch.cuda.current_device()) as clk:
        for _ in range(args.steps):
            t = time.perf_counter()
            outs, reps = binding.batch_all_edges(Gs, ells, **kw)
            times.append((time.perf_counter() - t) * 1e3)
    m = sum(g.m for g in gs)
    ms = statistics.mean(times)
    lens = [r["ell_global"] for r in reps]
    accuracy = None
    if refs is not None:
        errs = []
        for x, out, fut in zip(gs, outs, refs):
            kk, vals = fut.result()
            errs.append(float(np.max(np.abs(out[kk] - vals))))
        refs_ex.shutdown()
        bip = np.array([bool(x.meta.get("bipartite")) for x in gs])
        errs = np.array(errs)
        accuracy = {"graphs_checked": len(errs), "max_abs_err_worst_graph": float(errs.max()),
                    "max_abs_err_median_graph": float(np.median(errs)),
                    "graphs_above_eps": int(np.sum(errs > args.eps)),
                    "worst_lattice": float(errs[bip].max()) if bip.any() else None,
                    "worst_other": float(errs[~bip].max()) if (~bip).any() else None,
                    "oracle": "per graph: dense grounded-Laplacian inverse (n <= 5000, every edge) or 200 sampled "
                              "edges (sparse LU for lattices, CG otherwise), FP64, in a spawn pool on the host"}
    line = {"metric": "AESC edges/sec over a batch of 512 graphs (batched FP32, CUDA-graph launches)",
            "value": m / (ms / 1e3), "unit": UNIT, "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": ms, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic",
            "config": {"workload": "512 graphs, n log-uniform in [1000, 50000]: G(n, 8/(n-1)) LCC, "
                                   "Barabasi-Albert m=5, perturbed lattices, seeds 4..515",
                       "graphs": len(gs), "n_total": sum(g.n for g in gs), "m_total": m, "eps": args.eps,
                       "policy": "learned" if learned else "global (lattices: fixed)",
                       "lattice_length": None if learned else args.grid_ell,
                       "lattice_cap": args.batch_cap if learned else None,
                       "model": f"trained on {BATCH_TRAIN[0]}, 400 Adam steps" if learned else None,
                       "estimator": "end_corrected",
                       "lengths_min_max": [min(lens), max(lens)], "block_width": reps[0]["block_width"],
                       "source_hops": int(sum(r["source_hops"] for r in reps)),
                       "extension_rounds": reps[0]["extension_rounds"],
                       "hop_launches": reps[0]["hop_launches"], "generation_s": gen_s},
            "roofline": {"bound": "hbm", "achieved": reps[0]["hop_bytes"] / (reps[0]["propagate_ms"] / 1e3) / 1e9,
                         "peak": measured_peaks()[0], "unit": "GB/s", "note": "algorithmic bytes over the "
                         "propagation time (whole CUDA graph, not one kernel)"},
            "clocks": clk.summary(), "gpu_launches": int(reps[0]["launches"]), "accuracy": accuracy}
    line["roofline"]["frac"] = line["roofline"]["achieved"] / line["roofline"]["peak"]
    for G in Gs:
        G.close()
    if rank == 0:
        print(json.dumps(line), flush=True)


def run_caltau_arm(args, stream):
    """CalTau with omega eigenpairs on the device (Algorithm 1, Eq. 6-8) on a
    planted partition of 200,000 nodes (40 communities: 39 eigenvalues near 1),
    where Eq. 6 with lambda_2 alone asks hundreds of hops: the eigenpairs and
    CalTau calls timed on the host clock (they synchronise), sc_all_edges with
    the CalTau lengths by CUDA events after one warm-up; the lengths of Eq. 6
    reported beside them, not run."""
    import graphgen as gg
    import torch
    from paper_2305_16086_gb300 import Graph

    g = gg.workload("planted_200k")
    out = torch.empty(g.nnz, dtype=torch.float64, device="cuda")
    with Graph(g.row_ptr, g.col_idx, stream=stream) as G:
        t0 = time.perf_counter()
        _, _, rep = G.eigenpairs(omega=args.caltau_omega, allow_unconverged=True)
        t_eig = (time.perf_counter() - t0) * 1e3
        t0 = time.perf_counter()
        tau, ell = G.caltau(args.eps)
        t_ct = (time.perf_counter() - t0) * 1e3
        kw = dict(eps=args.eps, policy="caltau", precision=args.precision)
        G.all_edges(out=out, **kw)
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        _, _, r = G.all_edges(out=out, **kw)
        e1.record(stream)
        e1.synchronize()
        ms = e0.elapsed_time(e1)
        G.estimate_lambda(allow_unconverged=True)
        ell6, ps6, pe6 = G.truncation_length(args.eps)
    ps = np.maximum.reduceat(tau, g.row_ptr[:-1].astype(np.int64))
    return {"workload": "planted partition, 40 communities of 5000 nodes, internal degree 10, external 0.2, seed 6",
            "n": g.n, "m": g.m, "omega": args.caltau_omega, "pairs_taken": rep["used"],
            "lambda_rest": rep["lambda_rest"], "eigenpairs_ms": t_eig, "caltau_ms": t_ct,
            "all_edges_ms": ms, "value": g.m / (ms / 1e3), "unit": UNIT,
            "value_incl_eigenpairs_and_caltau": g.m / ((ms + t_eig + t_ct) / 1e3),
            "foster_mean_abs_error": ((g.n - 1) - r["foster_sum"]) / g.m,
            "mean_length": float(tau.mean()), "longest": int(ell), "source_hops": int(ps.sum()),
            "eq6": {"mean_length": float(pe6.mean()), "longest": int(ell6), "source_hops": int(ps6.sum()),
                    "note": "not run: the traversal at these lengths, for comparison"}}


def parse_args(argv=None):
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="ba_200k", choices=sorted(WORKLOADS) + ["batch_512"])
    ap.add_argument("--grid-ell", type=int, default=2201,
                    help="length of the lattices in batch_512 (no Eq. 6 length exists; 2201 keeps every lattice of "
                         "the batch within eps = 1e-3)")
    ap.add_argument("--eps", type=float, default=1e-3)
    ap.add_argument("--precision", default="fp32", choices=["fp64", "fp32", "bf16"])
    ap.add_argument("--policy", default="learned", choices=["learned", "global", "per_edge", "fixed"])
    ap.add_argument("--ell", type=int, default=0, help="length for --policy fixed")
    ap.add_argument("--estimator", default="plain", choices=["plain", "end_corrected"])
    ap.add_argument("--no-arms", action="store_true")
    ap.add_argument("--no-tgt-plus-arm", action="store_true", help="leave out the TGT+ arm (Algorithm 4)")
    ap.add_argument("--block-width", type=int, default=0)
    ap.add_argument("--rows-split", type=int, default=0)
    ap.add_argument("--heavy-threshold", type=int, default=0)
    ap.add_argument("--cpu-seconds", type=float, default=10.0)
    ap.add_argument("--check-edges", type=int, default=10000,
                    help="edges whose exact value the CPU baseline leg computes (CG) to report the error")
    ap.add_argument("--ref-step-seconds", type=float, default=8.0)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--caltau-arm", action="store_true",
                    help="also time CalTau with device eigenpairs (Algorithm 1) on a planted partition, n=200000")
    ap.add_argument("--caltau-omega", type=int, default=64)
    ap.add_argument("--mode", default="tgt", choices=["tgt", "tgt_plus"],
                    help="tgt: Algorithm 2; tgt_plus: Algorithm 4")
    ap.add_argument("--batch-cap", type=int, default=4095,
                    help="batch_512 with the learned policy: the lattices' longest length")
    ap.add_argument("--ell-cap", type=int, default=1023,
                    help="learned length on a bipartite graph: the longest length an edge may be extended to")
    ap.add_argument("--explicit-config", action="store_true",
                    help="keep --mode / --policy / --precision (/ --eps / --estimator) as given for the rmat_22 "
                         "and lattice_1000 workloads")
    args = ap.parse_args(argv)
    if args.workload == "rmat_22" and not args.explicit_config:
        # the R-MAT workload's configuration: TGT+ walks, learned lengths, BF16 storage from hop 8
        args.mode, args.policy, args.precision = "tgt_plus", "learned", "bf16"
    if args.workload == "lattice_1000" and not args.explicit_config:
        # the lattice's configuration: eps = 1e-2, learned lengths accepted by the tail estimate
        # (no bound exists on a bipartite graph), the end-corrected estimator, FP32 blocks
        args.eps, args.mode, args.policy = 1e-2, "tgt", "learned"
        args.estimator, args.precision = "end_corrected", "fp32"
    return args


def main():
    args = parse_args()
    if args.warmup < 3 and args.impl == "ours":
        print("warning: fewer than 3 warm-up steps", file=sys.stderr)
    world, rank, local = dist_setup()
    if args.impl == "reference":
        run_reference(args, world, rank)
        return
    if args.workload == "batch_512":
        run_batch(args, world, rank)
        return

    import torch

    import graphgen as gg
    from paper_2305_16086_gb300 import Graph, binding

    torch.cuda.set_device(local)
    pg = None
    if world > 1:
        import torch.distributed as dist

        dist.init_process_group("nccl")
        pg = dist
    g = WORKLOADS[args.workload]["make"](gg)
    stream = torch.cuda.current_stream()
    run_kw = dict(eps=args.eps, precision=args.precision, policy=args.policy, block_width=args.block_width,
                  rows_split=args.rows_split, heavy_threshold=args.heavy_threshold, ell_fixed=args.ell,
                  estimator=args.estimator, mode=args.mode, ell_cap=args.ell_cap)

    G = Graph(torch.from_numpy(g.row_ptr).cuda(), torch.from_numpy(g.col_idx).cuda(), stream=stream)
    bip = bool(G.info()["bipartite"])
    # the bound of Eq. 6 needs a converged lambda (its residual is the safety margin): an
    # unconverged estimate raises here and no value is reported. A fixed length, or any
    # length on a bipartite graph (lambda* = 1: no bound), does not use it.
    lambda_free = bip or args.policy == "fixed"
    lam = G.estimate_lambda(allow_unconverged=lambda_free)
    model = None
    if args.policy == "learned":
        # TGT+ certifies its truncation with eps / 2 (Algorithm 4's split): labels at eps / 2
        model = train_model(args.eps / 2 if args.mode == "tgt_plus" else args.eps, stream, args.workload)
        binding.mlp_load(G, model)
    out = torch.empty(g.nnz, dtype=torch.float64, device="cuda")
    flush = torch.empty(512 << 20, dtype=torch.uint8, device="cuda")  # > L2: evict between steps

    def barrier():
        if pg is not None:
            pg.barrier()
        torch.cuda.synchronize()

    for _ in range(args.warmup):
        G.all_edges(out=out, **run_kw)
    barrier()
    step_ms, reports = [], []
    with ClockSampler(torch.cuda.current_device()) as clk:
        barrier()
        for _ in range(args.steps):
            flush.zero_()
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            torch.cuda.nvtx.range_push("timed_step")
            e0.record(stream)
            _, _, rep = G.all_edges(out=out, time_kernels=True, **run_kw)
            e1.record(stream)
            torch.cuda.nvtx.range_pop()
            e1.synchronize()
            step_ms.append(e0.elapsed_time(e1))
            reports.append(rep)
        barrier()
    total_ms = max_over_ranks(pg, float(sum(step_ms)), "cuda")
    ms_per_step = total_ms / args.steps
    value = replica_value(world, g.m, ms_per_step)

    peak, peak_kind = measured_peaks()
    rep0 = reports[0]
    # every timed kernel class of the traversal; the roofline goes to the one with the most device time
    classes = {}
    for name in KERNEL_CLASSES:
        ms = sum(r["kernel_classes"][name]["ms"] for r in reports)
        nb = sum(r["kernel_classes"][name]["bytes"] for r in reports)
        nl = sum(r["kernel_classes"][name]["launches"] for r in reports)
        classes[name] = {"kernels": KERNEL_CLASSES[name], "ms_per_step": ms / args.steps,
                         "launches_per_step": nl / args.steps,
                         "share_of_step": ms / total_ms if total_ms > 0 else None,
                         "algorithmic_GBps": nb / (ms / 1e3) / 1e9 if ms > 0 and nb > 0 else None,
                         "_ms": ms, "_bytes": nb, "_launches": nl}
    top = max(classes, key=lambda k: classes[k]["_ms"])
    c = classes[top]
    achieved = c["_bytes"] / (c["_ms"] / 1e3) / 1e9 if c["_ms"] > 0 else 0.0
    config_key = f"{args.workload}/{args.precision}/B{rep0['block_width']}/v{rep0['rows_split']}/{top}"
    roofline = {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
                "traffic": recorded_traffic(config_key), "kernel": c["kernels"], "kernel_class": top,
                "peak_kind": peak_kind,
                "algorithmic_bytes_per_launch": c["_bytes"] / max(c["_launches"], 1),
                "avg_launch_us": c["_ms"] * 1e3 / max(c["_launches"], 1), "launches_timed": c["_launches"],
                "share_of_step": c["share_of_step"]}
    for v in classes.values():
        for k in ("_ms", "_bytes", "_launches"):
            v.pop(k)

    # end to end through the public API with host buffers: H2D of the CSR,
    # graph validation, eigenvalue bound, all edges, D2H of s_hat
    e2e = None
    if not args.no_e2e:
        rp_h = torch.from_numpy(g.row_ptr).pin_memory()
        ci_h = torch.from_numpy(g.col_idx).pin_memory()
        out_h = torch.empty(g.nnz, dtype=torch.float64).pin_memory()
        def e2e_pass(mark):
            with Graph(rp_h, ci_h, stream=stream) as Gh:
                mark("create_validate")
                Gh.estimate_lambda(allow_unconverged=lambda_free)
                mark("lanczos")
                if model is not None:
                    binding.mlp_load(Gh, model)
                mark("model_load")
                Gh.all_edges(out=out_h, **run_kw)
                mark("all_edges_d2h")

        e2e_ms, phases = timed_passes(e2e_pass, 2, min(args.steps, 3), torch.cuda.synchronize, barrier)
        e2e_step = max_over_ranks(pg, statistics.mean(e2e_ms), "cuda")
        e2e = {"value": replica_value(world, g.m, e2e_step), "unit": UNIT,
               "h2d_bytes_per_step": int(4 * (g.n + 1) + 4 * g.nnz), "d2h_bytes_per_step": int(8 * g.nnz),
               "ms_per_step": e2e_step,
               "includes": "graph create + validation + Lanczos + model load + features + all edges + D2H",
               "phases_ms_of_a_warmup_pass": phases}

    # comparison arms: TGT (traversal only) at the plain global length in FP32 and FP64
    # (one warm-up, one timed step each); on a bipartite graph the global length is the
    # empirical one (least odd length within eps on the sampled edges) in FP32
    arms = {}
    lat_ref = None
    if bip and rank == 0 and world == 1 and not args.no_cpu_baseline and args.check_edges > 0:
        lat_ref = lattice_reference(g, min(args.check_edges, 500))
    ours_host = out.cpu().numpy()
    if bip and not args.no_arms:
        ell_emp = None
        if lat_ref is not None:
            ell_emp = empirical_length(G, lat_ref, args.eps, args.ell_cap,
                                       dict(eps=args.eps, precision=args.precision, estimator="end_corrected"))
        if ell_emp is None:
            ell_emp = 105  # the least odd length within eps = 1e-2 on the 1000 x 1000 lattice's LU sample
        kw = dict(run_kw, policy="fixed", ell_fixed=ell_emp, estimator="end_corrected", mode="tgt")
        G.all_edges(out=out, **kw)
        barrier()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        _, _, r = G.all_edges(out=out, **kw)
        e1.record(stream)
        e1.synchronize()
        arms["global_emp_fp32"] = {"value": world * g.m / (e0.elapsed_time(e1) / 1e3), "unit": UNIT,
                                   "ms_per_step": e0.elapsed_time(e1), "source_hops": r["source_hops"],
                                   "ell": ell_emp,
                                   "ell_from": "least odd length within eps on the sampled edges (LU)"
                                   if lat_ref is not None else "fixed (no exact sample in this run)",
                                   "foster_mean_abs_error": ((g.n - 1) - r["foster_sum"]) / g.m}
        if lat_ref is not None:
            arms["global_emp_fp32"].update(errors_at(lat_ref, out.cpu().numpy()))
    elif not args.no_arms:
        arm_policy = "global" if args.policy == "learned" else args.policy
        for name, prec in ((f"{arm_policy}_fp32", "fp32"), (f"{arm_policy}_fp64", "fp64")):
            kw = dict(run_kw, policy=arm_policy, precision=prec, mode="tgt")
            G.all_edges(out=out, **kw)
            barrier()
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            _, _, r = G.all_edges(out=out, **kw)
            e1.record(stream)
            e1.synchronize()
            arms[name] = {"value": world * g.m / (e0.elapsed_time(e1) / 1e3), "unit": UNIT,
                          "ms_per_step": e0.elapsed_time(e1), "source_hops": r["source_hops"],
                          "foster_mean_abs_error": ((g.n - 1) - r["foster_sum"]) / g.m}
        if args.mode == "tgt" and not args.no_tgt_plus_arm:
            # Algorithm 4 (TGT+: traversal, switch test of Eq. 14 by the cost rule, Philox walks) at
            # the same eps, FP32 blocks, lengths of Eq. 6 at eps / 2
            kw = dict(run_kw, policy="global", precision="fp32", mode="tgt_plus")
            G.all_edges(out=out, **kw)
            barrier()
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            _, _, r = G.all_edges(out=out, **kw)
            e1.record(stream)
            e1.synchronize()
            arms["tgt_plus_fp32"] = {"value": world * g.m / (e0.elapsed_time(e1) / 1e3), "unit": UNIT,
                                     "ms_per_step": e0.elapsed_time(e1), "source_hops": r["source_hops"],
                                     "switch_after_hops": [r["tt_min"], r["tt_max"]], "walk_pairs": r["walks"],
                                     "walk_steps": r["walk_steps"], "switch_tests": r["switch_tests"],
                                     "switch_ms": r["switch_ms"], "walk_ms": r["walk_ms"],
                                     "ell_global": r["ell_global"],
                                     "foster_mean_abs_error": ((g.n - 1) - r["foster_sum"]) / g.m}

    if rank != 0:
        if pg is not None:
            pg.destroy_process_group()
        return
    cpu = None
    accuracy = None
    if not args.no_cpu_baseline and world == 1:
        cpu_ell = arms["global_emp_fp32"]["ell"] if "global_emp_fp32" in arms else rep0["ell_global"]
        cpu = cpu_baseline(g, cpu_ell, target_s=args.cpu_seconds)
        if lat_ref is not None:
            accuracy = dict(errors_at(lat_ref, ours_host),
                            oracle="FP64 sparse LU of the grounded Laplacian per sampled edge",
                            oracle_seconds=round(lat_ref["seconds"], 2), oracle_cores=lat_ref["cores"],
                            sample_seed=lat_ref["seed"])
        elif args.check_edges > 0:
            accuracy = exact_check(g, ours_host, args.check_edges)
    caltau_arm = run_caltau_arm(args, stream) if args.caltau_arm else None
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms_per_step, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": {"fp64": "f64", "fp32": "f32", "bf16": "bf16"}[args.precision],
        "data": "synthetic",
        "config": {"workload": WORKLOADS[args.workload]["desc"], "n": g.n, "m": g.m, "eps": args.eps,
                   "mode": args.mode, "policy": args.policy, "estimator": args.estimator,
                   "windowed": bool(rep0["windowed"]),
                   "precision": f"{args.precision} blocks, fp64 accumulation",
                   "batching": f"{rep0['slices']} block(s) of {rep0['block_width']} sources per launch, "
                               f"{rep0['blocks']} blocks",
                   "ell_global": rep0["ell_global"], "lambda_star": lam["lambda_star"],
                   "lambda_converged": bool(lam["converged"]), "lanczos_iterations": lam["iterations"],
                   "lambda_residuals": [lam["residual_plus"], lam["residual_minus"]],
                   "block_width": rep0["block_width"], "rows_split": rep0["rows_split"],
                   "slices": rep0["slices"], "l2": "working set > L2 and a 512 MB write between steps",
                   "parallelism": f"replicas x{world}"},
        "roofline": roofline, "kernel_classes": classes, "cpu_baseline": cpu, "e2e": e2e, "arms": arms,
        "learned": {"source_hops": rep0["source_hops"], "extension_rounds": rep0["extension_rounds"],
                    "edges_extended": rep0["edges_extended"], "max_tail_bound": rep0["max_tail_bound"],
                    "acceptance": "power-law tail estimate (uncertified: no bound exists at lambda* = 1)"
                    if rep0["uncertified"] else "a-posteriori bound (certified)",
                    "ell_cap": args.ell_cap if rep0["uncertified"] else None,
                    "model": f"trained on {TRAIN_GRAPHS.get(args.workload, DEFAULT_TRAIN)[0]}, 400 Adam steps"}
        if args.policy == "learned" else None,
        "tgt_plus": {"switch_after_hops": [rep0["tt_min"], rep0["tt_max"]], "walk_pairs": rep0["walks"],
                     "walk_steps": rep0["walk_steps"], "switch_tests": rep0["switch_tests"],
                     "switch_ms": rep0["switch_ms"], "walk_ms": rep0["walk_ms"]}
        if args.mode == "tgt_plus" else None,
        "caltau": caltau_arm,
        "clocks": clk.summary(), "gpu_launches": int(sum(r["launches"] for r in reports)),
        "foster_mean_abs_error": ((g.n - 1) - rep0["foster_sum"]) / g.m,
        "max_abs_err": accuracy["max_abs_err"] if accuracy else None,
        "mean_abs_err": accuracy["mean_abs_err"] if accuracy else None,
        "accuracy": accuracy,
    }
    print(json.dumps(line), flush=True)
    if pg is not None:
        pg.destroy_process_group()


if __name__ == "__main__":
    main()
