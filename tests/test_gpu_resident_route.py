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
