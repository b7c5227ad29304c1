"""The switch test's top-gamma list by counting (up to 256 candidates) and by
merged lists (up to 2,048, then the whole column): on a complete graph every
value but the source's ties, so a column of n nodes has about n candidates. Both
sides of each limit, and lists longer than the candidates, give what the scan of
every row gives, bit for bit."""
import numpy as np
import pytest

import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [24, 255, 256, 257, 258, 600, 2047, 2050])
def test_rank_and_merge_lists_equal_full_scan(cuda_lib, n, precision):
    from paper_2305_16086_gb300 import Graph

    g = gg.complete(n)
    with Graph(g.row_ptr, g.col_idx) as G:
        base = dict(eps=5e-3, mode="tgt_plus", seed=9, policy="fixed", ell_fixed=5, precision=precision, switch="paper",
                    gamma=16)
        s, _, rep = G.all_edges(**base)
        f, _, rep_f = G.all_edges(full_topgamma_scan=True, **base)
    assert rep["switch_tests"] > 0
    assert np.array_equal(s, f)
    for key in ("walks", "walk_steps", "tt_min", "tt_max", "switch_tests"):
        assert rep[key] == rep_f[key], key
