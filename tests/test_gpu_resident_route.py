"""Which sources of a small-degree graph run resident (report.resident_sources):
the value tests of the resident traversal compare it with the block kernels and
would pass if every source went there. A graph whose balls fit runs resident
whole; a ball larger than every list goes to the blocks; near a corner of the
same lattice it fits. The list bounds follow from 226 KB of shared memory: 28 bytes a
node with its adjacency (bipartite, FP32, four slots), 4 without it, ids below
65,000."""
import numpy as np
import pytest

import graphgen as gg
from test_gpu_resident import GRAPHS, _graph, _kings

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("ell,estimator", [(1, "plain"), (40, "end_corrected")])
def test_small_graphs_run_resident(cuda_lib, name, precision, ell, estimator):
    g = GRAPHS[name]()
    with _graph(g) as G:
        G.set_lambda(0.999, -0.999, 0.999)
        kw = dict(policy="fixed", ell_fixed=ell, precision=precision, estimator=estimator, bf16_from_hop=4)
        _, _, rep = G.all_edges(**kw)
        _, _, rep0 = G.all_edges(windows=False, **kw)
        _, _, rep1 = G.all_edges(windows=True, **kw)
    assert rep["resident_sources"] == g.n and rep["windowed"] == 1
    assert rep0["resident_sources"] == 0 and rep0["windowed"] == 0
    assert rep1["resident_sources"] == 0 and rep1["windowed"] == 1


@pytest.mark.parametrize("name", ["lattice", "renamed", "odd_cycle", "kings", "cube", "small"])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("ell", [63, 64, 331])
def test_runs_of_many_more_hops_than_levels(cuda_lib, name, precision, ell):
    """From 64 hops and four a level on the lists are in id order."""
    g = GRAPHS[name]()
    with _graph(g) as G:
        s, _, rep = G.all_edges(policy="fixed", ell_fixed=ell, precision=precision)
        s0, _, _ = G.all_edges(policy="fixed", ell_fixed=ell, precision=precision, windows=False)
    assert rep["resident_sources"] == g.n
    assert np.array_equal(s, s0)


@pytest.mark.parametrize("maker,ell,precision,share", [
    (lambda: gg.perturbed_grid(60, 140, 0.05, 5), 81, "fp32", "all"),    # 8,400 nodes, balls of half of them
    (lambda: gg.perturbed_grid(130, 131, 0.05, 5), 201, "fp32", "all"),  # 17,030 nodes: without the adjacency
    (lambda: gg.perturbed_grid(100, 111, 0.05, 5), 161, "fp64", "all"),
    (lambda: gg.perturbed_grid(260, 261, 0.05, 5), 401, "fp32", "some"),  # 67,860 nodes
    (lambda: _kings(90, 91), 121, "fp32", "some"),                        # two buffers: 4,400 nodes at most
    (lambda: gg.path(2600), 2301, "fp32", "none"),                        # 1,151 levels, bounds for 1,024
])
def test_large_balls_where_they_fit(cuda_lib, maker, ell, precision, share):
    from paper_2305_16086_gb300 import binding

    g = maker()
    ent = np.random.default_rng(2).integers(0, g.nnz, 150)
    nsrc = np.unique(np.concatenate([g.entry_rows()[ent], g.col_idx[ent]])).size
    with _graph(g) as G:
        _, rep = binding.some_edges(G, ent, policy="fixed", ell_fixed=ell, precision=precision)
    got = rep["resident_sources"]
    assert (got == nsrc) if share == "all" else (got == 0) if share == "none" else (0 < got < nsrc)


def test_batch_reports_each_graph(cuda_lib):
    from paper_2305_16086_gb300 import Graph, binding

    gs = [gg.perturbed_grid(20, 31, 0.05, 1), gg.barabasi_albert(500, 4, 2), gg.cycle(301), gg.path(2600)]
    Gs = [Graph(g.row_ptr, g.col_idx) for g in gs]
    try:
        _, reps = binding.batch_all_edges(Gs, [45, 9, 30, 2301], policy="fixed", precision="fp32")
    finally:
        for G in Gs:
            G.close()
    assert [r["resident_sources"] for r in reps] == [gs[0].n, 0, gs[2].n, 0]


def _regular(n, d, seed):
    """A random graph of degree d (even) without short cycles to speak of: d / 2 random Hamiltonian cycles."""
    rng = np.random.default_rng(seed)
    p = [rng.permutation(n) for _ in range(d // 2)]
    return gg.from_edges(n, np.concatenate(p), np.concatenate([np.roll(q, 1) for q in p]))


def _bipartite(n, d, seed):
    """A random bipartite graph of degree d: d random perfect matchings, renamed."""
    rng = np.random.default_rng(seed)
    h = n // 2
    name = rng.permutation(n)
    v = np.concatenate([h + rng.permutation(h) for _ in range(d)])
    return gg.largest_component(gg.from_edges(n, name[np.tile(np.arange(h), d)], name[v]))


@pytest.mark.parametrize("maker,ell,precision,resident", [
    (lambda: _bipartite(14000, 4, 2), 15, "fp32", False),  # most of the graph within 8 hops: blocks
    (lambda: _bipartite(14000, 4, 2), 15, "fp64", True),   # the same where a block's arithmetic is slow
    (lambda: gg.relabel(gg.perturbed_grid(130, 131, 0.05, 5), np.random.default_rng(1).permutation(17030)), 121,
     "fp32", True),
])
def test_balls_without_their_adjacency_by_cost(cuda_lib, maker, ell, precision, resident):
    """Balls past the classes that hold their adjacency: resident only where that
    is the faster form."""
    g = maker()
    kw = dict(policy="fixed", ell_fixed=ell, precision=precision)
    with _graph(g) as G:
        s, _, rep = G.all_edges(**kw)
        s0, _, _ = G.all_edges(windows=False, **kw)
    assert rep["resident_sources"] == (g.n if resident else 0)
    assert np.array_equal(s, s0)


def test_node_marks_are_taken_back(cuda_lib):
    """The class without the adjacency marks a ball's nodes and takes the marks
    back: calls of both precisions, of few sources and of many, and ones whose
    balls do not fit, leave nothing behind for the next."""
    from paper_2305_16086_gb300 import binding

    g = gg.perturbed_grid(130, 131, 0.05, 5)
    rng = np.random.default_rng(4)
    with _graph(g) as G:
        want = {}
        for p in ("fp32", "fp64"):
            want[p], _, _ = G.all_edges(policy="fixed", ell_fixed=141, precision=p, windows=False)
        for precision, count in (("fp32", 5), ("fp64", 300), ("fp32", 120), ("fp64", 4), ("fp32", 2000)):
            ent = rng.integers(0, g.nnz, count)
            q, rep = binding.some_edges(G, ent, policy="fixed", ell_fixed=141, precision=precision)
            nsrc = np.unique(np.concatenate([g.entry_rows()[ent], g.col_idx[ent]])).size
            assert rep["resident_sources"] == nsrc
            assert np.array_equal(q, want[precision][ent])
    # 67,860 nodes: in mid-lattice balls past the class, marks up to where they overflow
    g = gg.perturbed_grid(260, 261, 0.05, 5)
    mid = 130 * 261 + 130
    ent = g.row_ptr[mid:mid + 60].astype(np.int64)
    with _graph(g) as G:
        a, ra = binding.some_edges(G, ent, policy="fixed", ell_fixed=401, precision="fp32")
        b, rb = binding.some_edges(G, ent, policy="fixed", ell_fixed=201, precision="fp32")
        a0, _ = binding.some_edges(G, ent, policy="fixed", ell_fixed=401, precision="fp32", windows=False)
        b0, _ = binding.some_edges(G, ent, policy="fixed", ell_fixed=201, precision="fp32", windows=False)
    nsrc = np.unique(np.concatenate([g.entry_rows()[ent], g.col_idx[ent]])).size
    assert 0 < ra["resident_sources"] < nsrc and rb["resident_sources"] == nsrc
    assert np.array_equal(a, a0) and np.array_equal(b, b0)


@pytest.mark.parametrize("maker,ell,precision", [
    (lambda: _regular(9000, 8, 1), 7, "fp32"),       # no ball fits
    (lambda: _bipartite(14000, 4, 2), 15, "fp32"),   # balls that fit at a cost
    (lambda: gg.perturbed_grid(90, 100, 0.05, 5), 61, "fp32"),
])
def test_the_sample_of_a_whole_request_is_kept(cuda_lib, maker, ell, precision):
    """A repeated call launches what the first did but for the sample's launches
    (and the neighbour rows laid out once); another length, then the first again,
    and a query stay right."""
    from paper_2305_16086_gb300 import binding

    g = maker()
    kw = dict(policy="fixed", ell_fixed=ell, precision=precision)
    with _graph(g) as G:
        _, _, first = G.all_edges(**kw)
        s, _, again = G.all_edges(**kw)
        short, _, _ = G.all_edges(policy="fixed", ell_fixed=4, precision=precision)
        _, _, third = G.all_edges(**kw)
        ent = np.random.default_rng(3).integers(0, g.nnz, 300)
        q, _ = binding.some_edges(G, ent, **kw)
        s0, _, _ = G.all_edges(windows=False, **kw)
        short0, _, _ = G.all_edges(policy="fixed", ell_fixed=4, precision=precision, windows=False)
    assert again["launches"] == third["launches"] < first["launches"] - 1
    assert again["resident_sources"] == third["resident_sources"] == first["resident_sources"]
    assert np.array_equal(s, s0) and np.array_equal(q, s0[ent]) and np.array_equal(short, short0)


def _regular_with_path(n, length, seed):
    """A random graph of degree 8, one edge of it replaced by a long path."""
    c = _regular(n, 8, seed)
    e = c.edges()
    ids = np.concatenate([e[0, :1], n + np.arange(length), e[0, 1:]])
    return gg.from_edges(n + length, np.concatenate([e[1:, 0], ids[:-1]]), np.concatenate([e[1:, 1], ids[1:]]))


@pytest.mark.parametrize("maker,ell,precision,estimator,share,windows", [
    (lambda: _regular(9000, 8, 1), 7, "fp32", "plain", "none", False),   # balls of nearly the whole graph
    (lambda: _regular(9000, 8, 1), 9, "bf16", "end_corrected", "none", False),
    (lambda: _regular(18000, 8, 2), 7, "fp64", "plain", "none", False),  # sparse ends of a large graph's blocks
    # the path's sources run resident, then the blocks' shape is timed
    (lambda: _regular_with_path(9000, 900, 3), 9, "fp32", "end_corrected", "some", False),
    (lambda: _kings(90, 91), 121, "fp32", "end_corrected", "some", True),  # windows of 0.6 of the graph
])
def test_left_over_sources_take_the_better_blocks(cuda_lib, maker, ell, precision, estimator, share, windows):
    """Sources whose balls fit nowhere go to the blocks that a request without the
    resident form would take (hops 1-2 from masks, the last hop on the gather's
    rows), or to windows where they hold little of the graph, in a timed launch
    shape; the sums of the sources that ran before the timing stay as they are."""
    from paper_2305_16086_gb300 import binding

    g = maker()
    kw = dict(policy="fixed", ell_fixed=ell, precision=precision, estimator=estimator, bf16_from_hop=4)
    with _graph(g) as G:
        G.set_lambda(0.999, -0.999, 0.999)
        s, b, rep = G.all_edges(**kw)
        s0, b0, rep0 = G.all_edges(windows=False, **kw)
        ent = np.random.default_rng(3).integers(0, g.nnz, 40)  # few enough to go untimed
        q, rq = binding.some_edges(G, ent, **kw)
    got = rep["resident_sources"]
    assert (got == 0) if share == "none" else (0 < got < g.n)
    assert rep["windowed"] == (1 if got or windows else 0)
    kc = rep["kernel_classes"]
    assert (kc["mask_hop"]["launches"] > 0) == (not windows)
    assert (kc["last_hop"]["launches"] > 0) == (not windows)
    if share == "none":
        assert rq["kernel_classes"]["last_hop"]["launches"] > 0
    assert np.array_equal(s, s0) and np.array_equal(q, s0[ent])
    if b is not None:
        assert np.array_equal(b, b0)


def test_batches_of_graphs_that_do_not_run_resident(cuda_lib):
    """A member of which no source ran resident is left to the blocks in later
    batches of the same length and precision; others are tried again."""
    from paper_2305_16086_gb300 import Graph, binding

    gs = [_regular(6000, 8, 1), gg.perturbed_grid(20, 31, 0.05, 1), _regular(6000, 8, 2)]
    Gs = [Graph(g.row_ptr, g.col_idx) for g in gs]
    try:
        seen = []
        for ells, precision in (([9, 45, 9], "fp32"), ([9, 45, 9], "fp32"), ([3, 45, 9], "fp32"), ([9, 45, 9], "fp64")):
            out, reps = binding.batch_all_edges(Gs, ells, policy="fixed", precision=precision)
            for G, e, s in zip(Gs, ells, out):
                s0, _, _ = G.all_edges(policy="fixed", ell_fixed=e, precision=precision, windows=False)
                assert np.array_equal(s, s0)
            seen.append([r["resident_sources"] for r in reps])
    finally:
        for G in Gs:
            G.close()
    assert seen == [[0, 620, 0], [0, 620, 0], [6000, 620, 0], [0, 620, 0]]


@pytest.mark.parametrize("maker", [lambda: _regular(9000, 8, 1), lambda: _regular(6000, 4, 4)])
@pytest.mark.parametrize("policy", ["learned", "per_edge", "global"])
def test_lengths_by_policy(cuda_lib, maker, policy):
    """Lengths that differ by source, the learned length's records and its
    extension rounds through the resident form and its left-overs."""
    from paper_2305_16086_gb300 import binding

    g, t = maker(), gg.barabasi_albert(2500, 5, 21)
    init = np.random.default_rng(3).normal(0, 0.2, binding.MLP_PARAMS).astype(np.float32)
    with _graph(t) as Gt:
        Gt.estimate_lambda()
        model, _ = binding.mlp_train([Gt], init, epochs=60, lr=1e-2, eps=1e-3, precision="fp32")
    with _graph(g) as G:
        G.estimate_lambda()
        binding.mlp_load(G, model)
        for precision in ("fp32", "fp64"):
            kw = dict(policy=policy, eps=1e-3, precision=precision)
            s, b, rep = G.all_edges(record_tail=policy != "learned", **kw)
            s0, b0, rep0 = G.all_edges(record_tail=policy != "learned", windows=False, **kw)
            assert rep["extension_rounds"] == rep0["extension_rounds"]
            assert rep["edges_extended"] == rep0["edges_extended"]
            assert np.array_equal(s, s0) and (b is None or np.array_equal(b, b0))
