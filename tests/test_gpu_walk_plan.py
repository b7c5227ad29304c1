"""The walk phase's plan (chunks of 128 walk pairs per entry, planned per source
in tiles of 128 entries) at its edges: a wheel's hub row one entry short of,
at and past one and two tiles, entries with no more than one chunk and with
several, and launches whose last slots are empty. With FP64 blocks the GPU and
the oracle draw the same Philox walks: their numbers agree exactly and s_hat up
to the rounding of the sums (1e-10)."""
import numpy as np
import pytest

import graphgen as gg
from oracle import series, tgtplus, truncation

pytestmark = pytest.mark.gpu

CHUNK = TILE = 128


def _wheel(spokes):
    rim = np.arange(1, spokes + 1)
    return gg.from_edges(spokes + 1, np.concatenate([np.zeros_like(rim), rim]), np.concatenate([rim, np.roll(rim, -1)]))


@pytest.mark.parametrize("spokes", [TILE - 1, TILE, TILE + 1, 2 * TILE + 1])
def test_walk_plan_at_tile_and_chunk_edges(cuda_lib, spokes):
    from paper_2305_16086_gb300 import Graph

    g, eps, seed = _wheel(spokes), 0.02, 7
    with Graph(g.row_ptr, g.col_idx) as G:
        lam = G.estimate_lambda()["lambda_star"]
        s, _, rep = G.all_edges(eps=eps, mode="tgt_plus", policy="per_edge", precision="fp64", seed=seed,
                                switch="paper")
    tt = rep["tt_min"]
    tau = truncation.tau_entries(g.n, g.row_ptr, g.col_idx, eps / 2, lam)
    assert rep["tt_max"] == tt < tau.max()  # one launch, and walks were drawn
    half, counts = np.zeros(g.nnz), np.zeros(g.nnz, dtype=np.int64)
    for i in range(g.n):
        a, b = g.row_ptr[i], g.row_ptr[i + 1]
        gi, R, _ = tgtplus.tgt_plus_half(g.n, g.row_ptr, g.col_idx, i, tau[a:b], tt, eps, 1.0 / g.n, 10, seed, g.m)
        half[a:b], counts[a:b] = gi / g.degree[i], R
    assert counts.max() > CHUNK  # entries of several chunks
    assert rep["walks"] == counts.sum()
    assert rep["walk_steps"] == 2 * np.sum(counts * np.maximum(tau - tt, 0))
    assert np.max(np.abs(s - (half + half[series.reverse_entries(g.n, g.row_ptr, g.col_idx)]))) < 1e-10
