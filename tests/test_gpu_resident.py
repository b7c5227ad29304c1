"""The resident traversal (sources' balls in shared memory, graphs of degree at
most 8) against the block kernels on the whole graph: bit for bit, since both
sum a row's neighbours in CSR order and a row outside the ball is zero or is
never read. The graphs reach each form: one buffer (bipartite) and two, four and
eight neighbour slots, balls of every size class (the last with its adjacency
in global memory), balls too deep or too large for any of them, odd and even
lengths from 1 on, listed edges, and a batch that mixes both paths."""
import numpy as np
import pytest

import graphgen as gg

pytestmark = pytest.mark.gpu


def _graph(g):
    from paper_2305_16086_gb300 import Graph

    return Graph(g.row_ptr, g.col_idx)


def _kings(rows, cols):
    """A lattice with both diagonals: degree 8, odd cycles."""
    i = np.arange(rows * cols).reshape(rows, cols)
    u = np.concatenate([i[:, :-1].ravel(), i[:-1].ravel(), i[:-1, :-1].ravel(), i[:-1, 1:].ravel()])
    v = np.concatenate([i[:, 1:].ravel(), i[1:].ravel(), i[1:, 1:].ravel(), i[1:, :-1].ravel()])
    return gg.from_edges(rows * cols, u, v)


GRAPHS = {
    "lattice": lambda: gg.perturbed_grid(37, 41, 0.05, 3),
    "renamed": lambda: gg.relabel(gg.perturbed_grid(30, 50, 0.05, 4), np.random.default_rng(1).permutation(1500)),
    "odd_cycle": lambda: gg.cycle(1001),
    "path": lambda: gg.path(700),
    "kings": lambda: _kings(33, 47),
    "cube": lambda: gg.hypercube(8),
    "small": lambda: gg.grid(2, 3),
}


@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("ell,estimator", [(1, "plain"), (2, "plain"), (9, "end_corrected"), (40, "end_corrected")])
def test_equals_the_block_kernels(cuda_lib, name, precision, ell, estimator):
    g = GRAPHS[name]()
    kw = dict(policy="fixed", ell_fixed=ell, precision=precision, estimator=estimator, bf16_from_hop=4)
    with _graph(g) as G:
        G.set_lambda(0.999, -0.999, 0.999)
        s, b, rep = G.all_edges(**kw)
        s0, b0, rep0 = G.all_edges(windows=False, **kw)
    assert rep["source_hops"] == rep0["source_hops"] == g.n * (ell + (2 if estimator == "end_corrected" else 0))
    assert np.array_equal(s, s0)
    if b is not None:
        assert np.array_equal(b, b0)


@pytest.mark.parametrize("maker,ell,precision", [
    (lambda: gg.perturbed_grid(60, 140, 0.05, 5), 81, "fp32"),    # one CTA per SM
    (lambda: gg.perturbed_grid(130, 131, 0.05, 5), 201, "fp32"),  # adjacency in global memory
    (lambda: gg.perturbed_grid(100, 111, 0.05, 5), 161, "fp64"),
    (lambda: gg.perturbed_grid(260, 261, 0.05, 5), 401, "fp32"),  # 68k nodes: past every class
    (lambda: _kings(90, 91), 121, "fp32"),                        # two buffers: past every class
    (lambda: gg.path(2600), 2301, "fp32"),                        # deeper than the level bounds
])
def test_large_balls(cuda_lib, maker, ell, precision):
    g = maker()
    with _graph(g) as G:
        ent = np.random.default_rng(2).integers(0, g.nnz, 150)
        from paper_2305_16086_gb300 import binding

        kw = dict(policy="fixed", ell_fixed=ell, precision=precision)
        s, _ = binding.some_edges(G, ent, **kw)
        s0, _ = binding.some_edges(G, ent, windows=False, **kw)
    assert np.array_equal(s, s0)


def test_batch_of_both_paths(cuda_lib):
    from paper_2305_16086_gb300 import Graph, binding

    gs = [gg.perturbed_grid(20, 31, 0.05, 1), gg.barabasi_albert(500, 4, 2), gg.cycle(301), gg.gnp_lcc(600, 8.0, 3),
          gg.perturbed_grid(40, 25, 0.05, 4)]
    Gs = [Graph(g.row_ptr, g.col_idx) for g in gs]
    ells = [45, 9, 30, 11, 61]
    try:
        for G in Gs:
            G.set_lambda(0.999, -0.999, 0.999)
        out, reps = binding.batch_all_edges(Gs, ells, policy="fixed", precision="fp32", estimator="end_corrected")
        for G, e, s, rep in zip(Gs, ells, out, reps):
            s0, _, rep0 = G.all_edges(policy="fixed", ell_fixed=e, precision="fp32", estimator="end_corrected",
                                      windows=False)
            assert np.array_equal(s, s0) and rep["source_hops"] == rep0["source_hops"]
    finally:
        for G in Gs:
            G.close()
