"""Routes that a request takes by itself, on graphs that the resident traversal
does not take: windowed blocks on banded numberings (the rule at both sides of
its line), and TGT+ with hop 3 from X_2's sectors when two blocks exceed the L2's
share."""
import numpy as np
import pytest

import graphgen as gg
from oracle import series

pytestmark = pytest.mark.gpu

TOL64, TOL32 = 1e-12, 2e-6


def _graph(g):
    from paper_2305_16086_gb300 import Graph

    return Graph(g.row_ptr, g.col_idx)


def _band(n, width, seed):
    """A path and five random chords a node, none longer than `width`; one of that length."""
    rng = np.random.default_rng(seed)
    i = np.arange(n - 1)
    u = np.concatenate([i, rng.integers(0, n - width, 5 * n), [7]])
    v = np.concatenate([i + 1, u[n - 1:-1] + rng.integers(2, width + 1, 5 * n), [7 + width]])
    return gg.from_edges(n, u, v)


@pytest.mark.parametrize("estimator", ["plain", "end_corrected"])
def test_windows_on_a_banded_graph(cuda_lib, estimator):
    g = _band(6000, 17, 1)
    assert g.degree.max() > 8
    tau = 21
    k = np.random.default_rng(1).choice(g.nnz, 300, replace=False)
    rows = np.searchsorted(g.row_ptr, k, side="right") - 1
    ref, _ = series.series_entries(g.n, g.row_ptr, g.col_idx, tau, sources=np.unique(np.concatenate([rows, g.col_idx[k]])),
                                   end_corrected=estimator == "end_corrected")
    kw = dict(policy="fixed", ell_fixed=tau, estimator=estimator)
    with _graph(g) as G:
        G.set_lambda(0.999, -0.999, 0.999)
        for precision, tol in (("fp64", TOL64), ("fp32", TOL32)):
            s, b, rep = G.all_edges(precision=precision, **kw)
            s0, b0, rep0 = G.all_edges(precision=precision, windows=False, **kw)
            assert rep["windowed"] == 1 and rep["resident_sources"] == 0 and rep0["windowed"] == 0
            assert rep["hop_bytes"] < 0.7 * rep0["hop_bytes"]
            assert np.max(np.abs(s[k] - ref[k])) <= tol
            assert np.array_equal(s, s0) and (b is None or np.array_equal(b, b0))


@pytest.mark.parametrize("ell", [1, 2, 81, 82, 83, 84, 85, 86])
def test_where_the_windows_end(cuda_lib, ell):
    """The widest window, (ell + 1) / 2 hops and a row further on either side, against half the graph."""
    g = _band(6000, 33, 2)
    with _graph(g) as G:
        s, _, rep = G.all_edges(policy="fixed", ell_fixed=ell, precision="fp32")
        s0, _, _ = G.all_edges(policy="fixed", ell_fixed=ell, precision="fp32", windows=False)
    assert rep["windowed"] == (1 if 2 * (ell // 2 + 2) * 33 + 128 < g.n / 2 else 0)
    assert np.array_equal(s, s0)


@pytest.mark.parametrize("n,precision,slices", [(90000, "fp32", 2), (170000, "bf16", 2), (50000, "fp64", 1)])
def test_tgt_plus_hop_3_from_sectors(cuda_lib, n, precision, slices):
    """Blocks of 128 exceed the L2's share on these graphs and take hop 3 from X_2's
    sectors, twice as many blocks of 64 do not and run it in full. Both launch the
    same sources together, so they switch at the same hops and draw the same walks:
    the values are the same bit for bit."""
    g = gg.barabasi_albert(n, 4, 5)
    kw = dict(mode="tgt_plus", policy="global", eps=1e-3, precision=precision, bf16_from_hop=1, seed=3)
    with _graph(g) as G:
        G.estimate_lambda()
        s, _, rep = G.all_edges(block_width=128, max_slices=slices, **kw)
        s0, _, rep0 = G.all_edges(block_width=64, max_slices=2 * slices, **kw)
    assert rep["slices"] == slices and rep0["slices"] == 2 * slices
    assert rep["switch_tests"] == rep0["switch_tests"] > 0 and rep["walks"] == rep0["walks"] > 0
    kc, kc0 = rep["kernel_classes"], rep0["kernel_classes"]
    assert kc["sparse_hop"]["launches"] > 0 and kc0["sparse_hop"]["launches"] == 0
    assert kc["ball_hop"]["launches"] == 0
    assert np.array_equal(s, s0)
