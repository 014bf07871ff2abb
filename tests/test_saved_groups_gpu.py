"""The grouped form of spq_query_saved (blocks shared by component pair, then the witness of every
pair) gives, bit for bit, the distances and witnesses of the same pairs in small batches (a warp
per pair).  Unit weights make every second column tie (row by row search), weights 1..2 and random
ones few (column by column), in integers and in floats; blocks up to 500 wide, unreachable,
equal and out-of-range pairs, and a second slice of a batch above 4,194,304 pairs.  The launch
counts show which form ran."""

import numpy as np
import pytest
from _util import spq, torch_dev
from test_walk_records_gpu import _graph

import gen

pytestmark = pytest.mark.gpu

SLICE = 1 << 22


def _case(kind):
    if kind in ("ties", "holes", "float"):
        return _graph(kind)
    name, f32 = kind.split("_") if "_" in kind else (kind, "")
    if name == "unit":  # blocks of 4 x 13 vertices on a side
        g, (part, k) = gen.graphs.grid4(60, 50, wmax=1, seed=3), gen.partition.grid_blocks(60, 50, 13, 11)
    else:  # every vertex on the boundary, 500 to a component: 16 words of columns
        g = gen.graphs.grid4(100, 10, wmax=1 if name == "wideunit" else 9, seed=5)
        part, k = (np.arange(1000) // 100 % 2).astype(np.int32), 2
    return (gen.Graph(g.n, g.row_ptr, g.col, g.w.astype(np.float32), g.xy) if f32 else g), part, k


@pytest.mark.parametrize("kind,q", [("ties", 60_000), ("unit", 60_000), ("unit_f32", 60_000), ("holes", 300_000),
                                    ("float", 20_001), ("wide", 4096), ("wide_f32", 4097), ("wideunit", 4500),
                                    ("wideunit_f32", 4500)])
def test_grouped_witnesses(kind, q):
    m = spq()
    torch, dev = torch_dev()
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    g, part, k = _case(kind)
    h = m.spq_build(g.n, T(g.row_ptr), T(g.col), T(g.w), T(part), k)
    rng = np.random.default_rng(q)
    pairs = rng.integers(0, g.n, size=(q, 2)).astype(np.int32)
    pairs[5] = pairs[5, 0]
    pairs[11] = (-1, 3)
    pairs[q - 1] = (2, g.n)
    pairs = T(pairs)
    n0 = m.spq_kernel_launches()
    dist, saved = m.spq_query_saved(h, pairs)
    assert m.spq_kernel_launches() - n0 > 6  # keys, sort, items, blocks, witnesses
    with pytest.raises(m.SpqError):
        m.spq_query_status(h)  # the two pairs out of range
    for a in range(0, q, 4000):
        n0 = m.spq_kernel_launches()
        d, s = m.spq_query_saved(h, pairs[a : a + 4000].contiguous())
        assert m.spq_kernel_launches() - n0 == 1
        assert torch.equal(d.view(torch.int32), dist[a : a + 4000].view(torch.int32))
        assert torch.equal(s, saved[a : a + 4000])
    h.free()


def test_second_slice():
    m = spq()
    torch, dev = torch_dev()
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    g, part, k = _case("float")
    h = m.spq_build(g.n, T(g.row_ptr), T(g.col), T(g.w), T(part), k)
    q = SLICE + 5001
    pairs = torch.randint(0, g.n, (q, 2), dtype=torch.int32, device=dev, generator=torch.Generator(dev).manual_seed(1))
    dist, saved = m.spq_query_saved(h, pairs)
    for a, b in [(0, 30_000), (SLICE - 20_000, SLICE), (SLICE, q)]:
        for i in range(a, b, 4000):
            j = min(i + 4000, b)
            d, s = m.spq_query_saved(h, pairs[i:j].contiguous())
            assert torch.equal(d.view(torch.int32), dist[i:j].view(torch.int32))
            assert torch.equal(s, saved[i:j])
    m.spq_query_status(h)
    h.free()
