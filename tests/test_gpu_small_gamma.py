"""TGT+ on graphs with fewer nodes than gamma: the top-gamma list holds every
node, as the oracle's does."""
import numpy as np
import pytest

import graphgen as gg
from oracle import exact

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [4, 6, 9, 10, 11])
def test_fewer_nodes_than_gamma(cuda_lib, n):
    from paper_2305_16086_gb300 import Graph

    g = gg.complete(n)
    with Graph(g.row_ptr, g.col_idx) as G:
        base = dict(eps=0.05, mode="tgt_plus", seed=1, policy="fixed", ell_fixed=7, precision="fp64", switch="paper",
                    gamma=10)
        s, _, rep = G.all_edges(**base)
        f, _, rep_f = G.all_edges(full_topgamma_scan=True, **base)
    assert rep["switch_tests"] > 0 and np.array_equal(s, f) and rep["walks"] == rep_f["walks"]
    assert np.max(np.abs(s - exact.exact_dense(g.n, g.row_ptr, g.col_idx))) <= 0.05
