"""spq_query_saved of a large batch (grouped by component pair) gives, bit for bit, the
distances and witnesses that the same pairs give in small batches (a warp per pair):
integer weights with ties everywhere, float weights, unreachable, equal and out-of-range
pairs, components without and with more than 256 boundary vertices."""

import numpy as np
import pytest
from _util import spq, torch_dev
from test_walk_records_gpu import _graph

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["ties", "holes", "wide", "single", "float"])
@pytest.mark.parametrize("q", [4096, 20001])
def test_large_batches_give_the_same_witnesses(kind, q):
    m = spq()
    torch, dev = torch_dev()
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    g, part, k = _graph(kind)
    h = m.spq_build(g.n, T(g.row_ptr), T(g.col), T(g.w), T(part), k)
    rng = np.random.default_rng(q)
    pairs = rng.integers(0, g.n, size=(q, 2)).astype(np.int32)
    pairs[5] = pairs[5, 0]
    pairs[11] = (-1, 3)
    pairs[q - 1] = (2, g.n)
    pairs = T(pairs)
    dist, saved = m.spq_query_saved(h, pairs)
    with pytest.raises(m.SpqError):
        m.spq_query_status(h)  # the two pairs out of range
    for a in range(0, q, 1000):
        d, s = m.spq_query_saved(h, pairs[a : a + 1000].contiguous())
        assert torch.equal(d.view(torch.int32), dist[a : a + 1000].view(torch.int32))
        assert torch.equal(s, saved[a : a + 1000])
    h.free()
