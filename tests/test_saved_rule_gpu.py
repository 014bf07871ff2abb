"""Which batches spq_query_saved groups by component pair (needs a GPU): those whose pairs share
blocks.  A batch spread over so many component pairs that most groups hold one pair is answered
a warp per pair, in one launch."""

import numpy as np
import pytest
from _util import spq, torch_dev

import gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q,groups", [(4095, False), (50_000, False), (1_000_000, True)])
def test_spread_pairs_are_not_grouped(q, groups):
    m = spq()
    torch, dev = torch_dev()
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    g = gen.graphs.grid4(256, 256, wmax=100, seed=1)
    part, k = gen.partition.grid_blocks(256, 256, 16, 16)  # 65,536 ordered component pairs
    h = m.spq_build(g.n, T(g.row_ptr), T(g.col), T(g.w), T(part), k)
    pairs = T(np.random.default_rng(q).integers(0, g.n, size=(q, 2)).astype(np.int32))
    before = m.spq_kernel_launches()
    m.spq_query_saved(h, pairs)
    assert (m.spq_kernel_launches() - before > 1) == groups
    h.free()
