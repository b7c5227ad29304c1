"""Timed workloads of the library: what a user's program has it compute, over
the sizes, precisions, length policies and entry points that the configurations,
tests and benchmark of this repository use.

A case is a dict of plain values; ``kind`` names the entry point:

* ``all``      -- ``Graph.all_edges`` on a resident graph (lambda, model loaded);
* ``some``     -- ``some_edges``: a query for a few edges of a resident graph;
* ``batch``    -- ``batch_all_edges`` over resident graphs of uneven size;
* ``noalloc``  -- ``all_edges_noalloc`` on device CSR arrays;
* ``lambda``   -- ``Graph.estimate_lambda`` on a resident graph;
* ``whole``    -- host CSR in, host values out: creation, eigenvalue bound,
                  lengths and traversal in one call chain.

Graphs are synthetic and seeded (``graphgen``): tree + G(n, p), Barabasi-Albert,
perturbed lattices, R-MAT and the mixed batch family.
"""
import math

import numpy as np
import torch

import graphgen as gg
from paper_2305_16086_gb300 import Graph, binding

# hops a learned or a-priori length typically takes, where a case does not fix it (only for work())
TYPICAL = {"tree": 15, "ba": 6, "grid": 45, "rmat": 12, "gnp": 17}


def listed():
    return [
        # a few edges of a small resident graph: the smallest query a service answers, all latency
        {"name": "query_16_edges", "kind": "some", "family": "tree", "n": 400, "deg": 8.0, "count": 16,
         "precision": "fp32", "policy": "fixed", "ell": 15, "estimator": "plain"},
        # a small sparse graph in full precision, the method's plain form
        {"name": "tree_gnp_2000_fp64", "kind": "all", "family": "tree", "n": 2000, "deg": 10.0,
         "precision": "fp64", "policy": "fixed", "ell": 15, "estimator": "plain"},
        # a caller that may not allocate device memory (a serving arena)
        {"name": "noalloc_4001_fp64", "kind": "noalloc", "family": "tree", "n": 4001, "deg": 8.0, "ell": 13},
        # one-shot use: a small social graph from host arrays to host values
        {"name": "whole_ba_5000", "kind": "whole", "family": "ba", "n": 5000, "deg": 5, "precision": "fp32",
         "policy": "global", "eps": 1e-3, "estimator": "plain"},
        # the eigenvalue bound of a power-law graph, preprocessing of every new graph
        {"name": "lambda_ba_100k", "kind": "lambda", "family": "ba", "n": 100000, "deg": 10},
        # a power-law graph in full precision at one length
        {"name": "ba_20k_fp64", "kind": "all", "family": "ba", "n": 20011, "deg": 10, "precision": "fp64",
         "policy": "fixed", "ell": 7, "estimator": "plain"},
        # the benchmark's workload: power-law graph, lengths from the trained model, certified
        {"name": "ba_200k_learned", "kind": "all", "family": "ba", "n": 200000, "deg": 10, "precision": "fp32",
         "policy": "learned", "eps": 1e-3, "estimator": "plain"},
        # traversal completed by random walks
        {"name": "ba_40k_walks", "kind": "all", "family": "ba", "n": 40000, "deg": 10, "precision": "fp32",
         "policy": "global", "eps": 1e-3, "estimator": "plain", "mode": "tgt_plus"},
        # skewed degrees: walks at learned lengths, bf16 storage of the late hops
        {"name": "rmat_14_composite", "kind": "all", "family": "rmat", "n": 1 << 14, "deg": 16, "precision": "bf16",
         "policy": "learned", "eps": 1e-3, "estimator": "plain", "mode": "tgt_plus"},
        # a road-like lattice, learned lengths accepted by the tail estimate and extended
        {"name": "lattice_400_learned", "kind": "all", "family": "grid", "n": 160000, "cols": 400,
         "precision": "fp32", "policy": "learned", "eps": 1e-2, "cap": 1023, "estimator": "end_corrected"},
        # a long strip of the same at one given length
        {"name": "strip_150x613_fixed", "kind": "all", "family": "grid", "n": 91950, "cols": 150,
         "precision": "fp32", "policy": "fixed", "ell": 67, "estimator": "end_corrected"},
        # many graphs of uneven size in one call, the three families in turn, slow lattices at a long length
        {"name": "batch_24_mixed", "kind": "batch", "count": 24, "nmin": 1000, "nmax": 6000, "precision": "fp32",
         "ell": 15, "grid_ell": 1001, "estimator": "end_corrected"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["some", "tree", "ba", "ba", "walks", "rmat", "grid", "grid", "batch", "noalloc", "lambda",
                       "whole"])
    if kind == "some":
        return {"kind": "some", "family": rng.choice(["tree", "ba"]), "n": _log(rng, 300, 20000),
                "deg": rng.choice([5, 8, 10]), "count": _log(rng, 1, 500),
                "precision": rng.choice(["fp64", "fp32"]), "policy": "fixed", "ell": rng.choice([5, 7, 11, 15]),
                "estimator": "plain"}
    if kind == "tree":
        return {"kind": "all", "family": "tree", "n": _log(rng, 300, 20000), "deg": rng.choice([6, 8, 10]),
                "precision": rng.choice(["fp64", "fp32"]), "policy": "fixed", "ell": rng.choice([9, 13, 15, 21]),
                "estimator": rng.choice(["plain", "end_corrected"])}
    if kind == "ba":
        return {"kind": "all", "family": "ba", "n": _log(rng, 3000, 150000), "deg": rng.choice([5, 6, 10]),
                "precision": "fp32", "policy": rng.choice(["learned", "global", "per_edge"]), "eps": 1e-3,
                "estimator": "plain"}
    if kind == "walks":
        return {"kind": "all", "family": "ba", "n": _log(rng, 3000, 60000), "deg": rng.choice([6, 10]),
                "precision": rng.choice(["fp64", "fp32"]) if rng.random() < 0.3 else "fp32", "policy": "global",
                "eps": rng.choice([1e-3, 2e-3]), "estimator": "plain", "mode": "tgt_plus"}
    if kind == "rmat":
        plus = rng.random() < 0.5
        return {"kind": "all", "family": "rmat", "n": 1 << rng.choice([12, 13, 14, 15]), "deg": rng.randint(9, 16),
                "precision": rng.choice(["fp32", "bf16"]), "policy": "learned" if plus else "global", "eps": 1e-3,
                "estimator": "plain", "mode": "tgt_plus" if plus else "tgt"}
    if kind == "grid":
        cols = rng.randint(60, 400)
        n = cols * max(60, _log(rng, 6000, 160000) // cols)
        learned = rng.random() < 0.5
        c = {"kind": "all", "family": "grid", "n": n, "cols": cols, "precision": rng.choice(["fp32", "fp32", "fp64"]),
             "policy": "learned" if learned else "fixed", "estimator": "end_corrected"}
        if c["precision"] == "fp64" and n > 60000:
            c["precision"] = "fp32"
        c.update({"eps": 1e-2, "cap": 1023} if learned else {"ell": rng.choice([21, 45, 67, 105])})
        return c
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(3, 24), "nmin": 500, "nmax": _log(rng, 2000, 6000),
                "precision": "fp32", "ell": rng.choice([9, 15, 21]), "grid_ell": rng.choice([201, 501, 1001]),
                "estimator": "end_corrected"}
    if kind == "noalloc":
        return {"kind": "noalloc", "family": "tree", "n": _log(rng, 300, 12000), "deg": rng.choice([6, 8, 10]),
                "ell": rng.choice([1, 5, 9, 13])}
    if kind == "lambda":
        return {"kind": "lambda", "family": rng.choice(["tree", "ba"]), "n": _log(rng, 1000, 100000),
                "deg": rng.choice([6, 8, 10])}
    return {"kind": "whole", "family": "ba", "n": _log(rng, 1000, 12000), "deg": rng.choice([5, 6]),
            "precision": "fp32", "policy": "global", "eps": 1e-3, "estimator": "plain"}


def _renamed(g, seed):
    """The same structure under another random numbering (the families whose edge count varies by seed)."""
    return gg.relabel(g, np.random.default_rng(seed).permutation(g.n))


def _graph(case, seed):
    f, n = case["family"], case["n"]
    if f == "tree":
        return _renamed(gg.tree_plus_gnp(n, float(case["deg"]), 3), seed)
    if f == "ba":
        return gg.barabasi_albert(n, int(case["deg"]), seed)
    if f == "grid":
        return gg.perturbed_grid(n // case["cols"], case["cols"], 0.05, seed)
    if f == "rmat":
        return _renamed(gg.rmat(n.bit_length() - 1, int(case["deg"]), seed=5), seed)
    raise KeyError(f)


def _batch(case, seed):
    """The mixed family at the sizes of one batch: a draw of its own of each graph for every seed."""
    out = []
    for i, g in enumerate(gg.batch_graphs(case["count"], case["nmin"], case["nmax"], base_seed=4)):
        if i % 3 == 0:
            g = _renamed(g, seed + i)
        elif i % 3 == 1:
            g = gg.barabasi_albert(g.n, 5, seed + i)
        else:
            r = int(math.ceil(math.sqrt(g.n)))  # the family's lattices: r x r or r x (r - 1) nodes
            g = gg.perturbed_grid(r, g.n // r, 0.05, seed + i)
        out.append(g)
    return out


def _model(case):
    """The length model, trained on a smaller graph of the family (fixed seeds)."""
    f = case["family"]
    if f == "ba":
        t = gg.barabasi_albert(3000, int(case["deg"]), 101)
    elif f == "rmat":
        t = gg.rmat(11, int(case["deg"]), seed=15)
    else:
        t = gg.perturbed_grid(60, 60, 0.05, 102)
    bip = f == "grid"
    eps = case["eps"] * (0.5 if case.get("mode") == "tgt_plus" else 1.0)
    init = np.random.default_rng(0).normal(0.0, 0.2, binding.MLP_PARAMS).astype(np.float32)
    with Graph(t.row_ptr, t.col_idx) as G:
        G.estimate_lambda(allow_unconverged=True)
        model, _ = binding.mlp_train([G], init, epochs=300, lr=1e-2, eps=eps, precision="fp32",
                                     ell_cap=255 if bip else 0)
    return model


def _options(case):
    kw = {"precision": case["precision"], "policy": case["policy"], "estimator": case["estimator"],
          "mode": case.get("mode", "tgt"), "eps": case.get("eps", 1e-3)}
    if case["policy"] == "fixed":
        kw["ell_fixed"] = case["ell"]
    if "cap" in case:
        kw["ell_cap"] = case["cap"]
    return kw


def _entries(case, nnz, seed):
    return np.random.default_rng(seed + 1).integers(0, nnz, size=case["count"]).astype(np.int64)


def _ells(case, gs):
    return [case["grid_ell"] if g.meta.get("bipartite") else case["ell"] for g in gs]


def prepare(case, seed):
    dev = torch.device("cuda")
    kind = case["kind"]
    if kind == "batch":
        gs = _batch(case, seed)
        Gs = [Graph(g.row_ptr, g.col_idx) for g in gs]
        for G in Gs:  # the tail bound of the end-corrected estimator
            G.set_lambda(0.999999, -0.999999, 0.999999)
        return {"case": case, "graphs": Gs, "ells": _ells(case, gs),
                "outs": [torch.empty(g.nnz, dtype=torch.float64, device=dev) for g in gs]}
    g = _graph(case, seed)
    if kind == "whole":
        return {"case": case, "row_ptr": g.row_ptr, "col_idx": g.col_idx}
    if kind == "noalloc":
        return {"case": case, "row_ptr": torch.from_numpy(g.row_ptr).to(dev),
                "col_idx": torch.from_numpy(g.col_idx).to(dev),
                "out": torch.empty(g.nnz, dtype=torch.float64, device=dev)}
    st = {"case": case, "graph": Graph(g.row_ptr, g.col_idx)}
    if kind == "lambda":
        return st
    st["options"] = _options(case)
    if case["estimator"] == "end_corrected" and case["policy"] == "fixed":
        st["graph"].set_lambda(0.999999, -0.999999, 0.999999)  # the caller's bound, for the tail column
    elif case["policy"] != "fixed":
        st["graph"].estimate_lambda(allow_unconverged=True)
    if case["policy"] == "learned":
        binding.mlp_load(st["graph"], _model(case))
    if kind == "some":
        st["entries"] = _entries(case, g.nnz, seed)
        st["out"] = torch.empty(case["count"], dtype=torch.float64, device=dev)
        return st
    st["out"] = torch.empty(g.nnz, dtype=torch.float64, device=dev)
    if case.get("mode", "tgt") == "tgt" and (case["estimator"] == "end_corrected" or case["policy"] == "learned"):
        st["bound"] = torch.zeros(g.nnz, dtype=torch.float64, device=dev)
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "all":
        s, b, _ = state["graph"].all_edges(out=state["out"], tail_bound=state.get("bound"), **state["options"])
        return [s] if b is None else [s, b]
    if kind == "some":
        s, _ = binding.some_edges(state["graph"], state["entries"], out=state["out"], **state["options"])
        return [s]
    if kind == "batch":
        outs, _ = binding.batch_all_edges(state["graphs"], state["ells"], state["outs"], precision=case["precision"],
                                          policy="fixed", estimator=case["estimator"])
        return outs
    if kind == "noalloc":
        return [binding.all_edges_noalloc(state["row_ptr"], state["col_idx"], case["ell"], state["out"])]
    if kind == "lambda":
        lam = state["graph"].estimate_lambda(allow_unconverged=True)
        return [np.array([lam["lambda_plus"], lam["lambda_minus"], lam["lambda_star"]])]
    with Graph(state["row_ptr"], state["col_idx"]) as G:
        lam = G.estimate_lambda(allow_unconverged=True)
        s, _, _ = G.all_edges(**_options(case))
    return [s, np.array([lam["lambda_plus"], lam["lambda_minus"], lam["lambda_star"]])]


# ---- work: the traversal's arithmetic with the walk's own support ---------------------------------
def _size(family, n, deg, cols):
    if family == "grid":
        return n, int(2 * 1.9 * n)
    return n, int(n * (2 * deg if family in ("ba", "rmat") else deg))


def _support(family, n, nnz, ell):
    """CSR entries next to the nodes a walk of ell hops can reach and return from."""
    if family == "grid":
        return min(nnz, 4.0 * (2 * ell * ell + 1) / 2)
    return min(nnz, (nnz / n) ** (ell + 1))


def _traversal(family, n, nnz, ell, sources=None):
    per = sum(2.0 * _support(family, n, nnz, min(h, ell - h + 1)) for h in range(1, ell + 1))
    return per * (n if sources is None else sources)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        total_b = total_f = 0.0
        for i in range(case["count"]):
            n = math.exp(0.5 * (math.log(case["nmin"]) + math.log(case["nmax"])))
            fam = ("gnp", "ba", "grid")[i % 3]
            n, nnz = _size(fam, int(n), 8 if fam == "gnp" else 5, 0)
            total_b += 4 * (n + 1) + 12.0 * nnz
            total_f += _traversal(fam, n, nnz, case["grid_ell"] if fam == "grid" else case["ell"])
        return {"bytes": total_b, "flops": total_f}
    fam = case["family"]
    n, nnz = _size(fam, case["n"], case.get("deg", 4), case.get("cols", 0))
    csr = 4.0 * (n + 1) + 4.0 * nnz
    if kind == "lambda":
        steps = 300  # one product and one sweep over the basis a step
        return {"bytes": csr + 8.0 * n, "flops": steps * 2.0 * nnz + 2.0 * steps * steps * n}
    ell = case.get("ell", TYPICAL[fam])
    if kind == "some":
        return {"bytes": csr + 16.0 * case["count"],
                "flops": _traversal(fam, n, nnz, ell, min(n, 2 * case["count"]))}
    return {"bytes": csr + 8.0 * nnz * (2 if case.get("estimator") == "end_corrected" else 1),
            "flops": _traversal(fam, n, nnz, ell)}


# ---- the same values in 64 bits, from the definition ---------------------------------------------
def _series(row_ptr, col_idx, ell, end_corrected):
    """Per CSR entry: S_ell = sum over l <= ell of the hop terms of both half sums, with t_{ell+1}/2
    for the end-corrected estimator, and t_{ell+1} + t_{ell+2}. By blocks of source columns."""
    dev = torch.device("cuda")
    n = len(row_ptr) - 1
    rp = torch.from_numpy(np.asarray(row_ptr)).to(dev).long()
    ci = torch.from_numpy(np.asarray(col_idx)).to(dev).long()
    deg = (rp[1:] - rp[:-1]).double()
    rows = torch.repeat_interleave(torch.arange(n, device=dev), rp[1:] - rp[:-1])
    P = torch.sparse_csr_tensor(rp, ci, (1.0 / deg)[rows], size=(n, n))
    hops = ell + (2 if end_corrected else 0)
    half = torch.zeros(ci.numel(), dtype=torch.float64, device=dev)
    t1, t2 = torch.zeros_like(half), torch.zeros_like(half)
    width = max(32, min(4096, (1 << 27) // n))
    for c0 in range(0, n, width):
        c1 = min(n, c0 + width)
        X = torch.zeros(n, c1 - c0, dtype=torch.float64, device=dev)
        X[torch.arange(c0, c1, device=dev), torch.arange(c1 - c0, device=dev)] = 1.0
        a, b = int(rp[c0]), int(rp[c1])
        src, nbr = rows[a:b], ci[a:b]
        for h in range(hops + 1):
            if h:
                X = torch.sparse.mm(P, X)
            term = (X[src, src - c0] - X[nbr, src - c0]) / deg[src]
            if h <= ell:
                half[a:b] += term
            elif h == ell + 1:
                t1[a:b] = term
            else:
                t2[a:b] = term
    key = rows * n + ci
    rev = torch.searchsorted(key, ci * n + rows)
    s = half + half[rev]
    t1, t2 = t1 + t1[rev], t2 + t2[rev]
    return (s + 0.5 * t1 if end_corrected else s), t1 + t2


def exact(case, seed):
    kind = case["kind"]
    if kind in ("lambda", "whole"):
        return None  # the residual in lambda_star belongs to the iteration
    if kind == "batch":
        gs = _batch(case, seed)
        if sum(g.n * g.nnz * float(e) for g, e in zip(gs, _ells(case, gs))) > 2.5e12:
            return None
        return [_series(g.row_ptr, g.col_idx, e, True)[0] for g, e in zip(gs, _ells(case, gs))]
    if kind != "noalloc" and case["policy"] != "fixed":
        return None  # lengths from the estimate or the model
    g = _graph(case, seed)
    if g.n * g.nnz * float(case["ell"] + 2) > 2.5e12:
        return None
    end = case.get("estimator") == "end_corrected"
    s, q = _series(g.row_ptr, g.col_idx, case["ell"], end)
    if kind == "some":
        return [s[torch.from_numpy(_entries(case, g.nnz, seed)).to(s.device)]]
    if end:
        return [s, q / (2.0 * (1.0 - 0.999999))]
    return [s]
