"""The work lists of the ball hop (hop L - 1 on the sources' two-hop balls): one
array per slice with the pairs of the rows of 1, 2, 3-4 and 5-8 chunks end to
end, sixteen for a row at most. Values against the windowed blocks bit for bit on
degrees of every kind with several slices to a launch, and the device memory
that a call takes."""
import numpy as np
import pytest

import graphgen as gg

pytestmark = pytest.mark.gpu


def _graph(g):
    from paper_2305_16086_gb300 import Graph

    return Graph(g.row_ptr, g.col_idx)


def _stairs(n, seed):
    """Degrees in stairs: a ring, and rows of about 30, 33, 60, 65, 120, 130, 250 and 300 random neighbours."""
    rng = np.random.default_rng(seed)
    i = np.arange(n)
    u, v = [i], [(i + 1) % n]
    for k, d in enumerate((28, 31, 58, 63, 118, 128, 248, 300)):
        rows = np.arange(40 * k, 40 * k + 40)
        u.append(np.repeat(rows, d))
        v.append(rng.integers(400, n, 40 * d))
    return gg.from_edges(n, np.concatenate(u), np.concatenate(v))


@pytest.mark.parametrize("maker", [lambda: _stairs(17000, 1), lambda: gg.rmat(13, 8)])
@pytest.mark.parametrize("precision,width,slices", [("fp32", 128, 3), ("fp32", 32, 5), ("fp64", 64, 2), ("bf16", 128, 4)])
@pytest.mark.parametrize("ell", [4, 6])
def test_every_kind_of_row_with_several_slices(cuda_lib, maker, precision, width, slices, ell):
    g = maker()
    kw = dict(policy="fixed", ell_fixed=ell, precision=precision, bf16_from_hop=1, block_width=width)
    with _graph(g) as G:
        s, _, rep = G.all_edges(sparse_hops=True, max_slices=slices, **kw)
        s0, _, _ = G.all_edges(windows=True, **kw)
    assert rep["slices"] == slices and rep["kernel_classes"]["ball_hop"]["launches"] > 0
    assert np.array_equal(s, s0)


def test_memory_of_a_sparse_call(cuda_lib):
    """32 slices of 128 columns on 20,000 nodes: beside the two blocks the lists
    take 16 words a node and slice, the masks eight, the rest a few."""
    import torch

    g = gg.barabasi_albert(20000, 6, 3)
    slices, width = 32, 128
    kw = dict(policy="fixed", ell_fixed=7, precision="fp32", block_width=width, max_slices=slices)
    with _graph(gg.barabasi_albert(17000, 6, 3)) as G:  # the kernels' code and the context's own memory
        G.all_edges(**kw)
    with _graph(g) as G:
        before = torch.cuda.mem_get_info()[0]
        _, _, rep = G.all_edges(**kw)
        taken = before - torch.cuda.mem_get_info()[0]
    assert rep["slices"] == slices and rep["kernel_classes"]["ball_hop"]["launches"] > 0
    nodes = slices * g.n
    blocks, lists, masks = 2 * nodes * width * 4, 16 * 4 * nodes, 2 * nodes * width // 8
    rest = 8 * nodes + 100 * g.nnz + (64 << 20)  # row lists, sector masks; per entry; 2 MB a buffer
    assert taken <= blocks + lists + masks + rest, (taken, blocks, lists, masks, rest)
