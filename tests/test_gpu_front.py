"""The sparse hops a block takes by itself (graphs of at least 16,384 nodes, sparse
X_2) against the windowed blocks, which run every hop in full: bit for bit. Rows of
one chunk, of up to eight and of many (heavy rows, cut into chunks), sources whose
two-hop balls are small and hubs whose balls are whole graphs, lengths with and
without full hops between the sparse ones, and the records of the learned length."""
import numpy as np
import pytest

import graphgen as gg

pytestmark = pytest.mark.gpu


def _graph(g):
    from paper_2305_16086_gb300 import Graph

    return Graph(g.row_ptr, g.col_idx)


def _hub_ring():
    """A ring of 20,000 nodes with chords and one node joined to every 20th: degrees 3 to 1,000."""
    i = np.arange(20000)
    return gg.from_edges(20000, np.concatenate([i, i[::2], np.zeros(1000, np.int64)]),
                         np.concatenate([(i + 1) % 20000, (i[::2] + 7919) % 20000, i[::20]]))


@pytest.mark.parametrize("maker", [lambda: gg.barabasi_albert(17011, 6, 3), _hub_ring,
                                   lambda: gg.tree_plus_gnp(16500, 9.0, 2)])
@pytest.mark.parametrize("precision,ell,width", [("fp32", 5, 0), ("fp32", 6, 128), ("fp64", 5, 0), ("fp64", 9, 128),
                                                 ("fp32", 4, 32), ("bf16", 7, 32), ("bf16", 7, 64)])
def test_equals_windowed_full_hops(cuda_lib, maker, precision, ell, width):
    from paper_2305_16086_gb300 import binding

    g = maker()
    ent = np.concatenate([np.random.default_rng(4).integers(0, g.nnz, 400), np.arange(40)])
    kw = dict(policy="fixed", ell_fixed=ell, precision=precision, bf16_from_hop=1, block_width=width, time_kernels=True)
    with _graph(g) as G:
        s, rep = binding.some_edges(G, ent, **kw)
        s0, _ = binding.some_edges(G, ent, windows=True, **kw)
    assert rep["kernel_classes"]["ball_hop"]["launches"] > 0
    assert np.array_equal(s, s0)


def test_learned_records(cuda_lib):
    from paper_2305_16086_gb300 import binding

    g, t = gg.barabasi_albert(17000, 5, 7), gg.barabasi_albert(3000, 5, 8)
    init = np.random.default_rng(0).normal(0.0, 0.2, binding.MLP_PARAMS).astype(np.float32)
    with _graph(t) as Gt:
        Gt.estimate_lambda()
        model, _ = binding.mlp_train([Gt], init, epochs=60, lr=1e-2, eps=1e-3, precision="fp32")
    with _graph(g) as G:
        G.estimate_lambda()
        binding.mlp_load(G, model)
        s, _, rep = G.all_edges(policy="learned", precision="fp32", time_kernels=True)
        s0, _, _ = G.all_edges(policy="learned", precision="fp32", windows=True)
    assert rep["kernel_classes"]["ball_hop"]["launches"] > 0
    assert np.array_equal(s, s0)
