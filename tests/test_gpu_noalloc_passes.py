"""sc_all_edges_noalloc on graphs whose sources take several passes through the
static array (several blocks of 32 side by side in each): the later passes reuse
both ping-pong buffers with the earlier ones' values in them, the last one has
fewer blocks and its last block fewer sources. Against sc_all_edges (FP64) and
the FP64 series oracle, one graph straight after another."""
import numpy as np
import pytest

import graphgen as gg
from test_zz_no_alloc import TOL64, _noalloc, _reference

pytestmark = pytest.mark.gpu

SCRATCH = 64 << 20


@pytest.mark.parametrize("ells", [(1, 2), (2, 4), (4, 1), (7, 5)])
def test_several_passes(cuda_lib, ells):
    import torch

    from oracle import series

    stream = torch.cuda.current_stream()
    graphs = [gg.tree_plus_gnp(4001, 8.0, 3), gg.barabasi_albert(5003, 4, 2)]
    for g, ell in zip(graphs, ells):
        blocks = SCRATCH // (2 * 8 * 32 * g.n)  # at most, in a pass
        assert g.n > 2 * 32 * blocks and g.n % 32 and (g.n // 32 + 1) % blocks
        got = _noalloc(cuda_lib, g, ell, stream)
        assert np.max(np.abs(got - _reference(g, ell))) <= TOL64
        ref, _ = series.series_entries(g.n, g.row_ptr, g.col_idx, ell)
        assert np.max(np.abs(got - ref)) <= TOL64
