"""Large batches of path walks go by the hop and slot records made once per call, small
ones search every hop: both take the same moves.  Paths are compared vertex for vertex with
the same pairs asked in small batches, gradients with the small batches' sum.

Tolerance of the gradients: every slot's value is a sum of at most q float32 terms of
magnitude up to max|g|, in another order: |difference| <= 2 q 2^-24 sum|g| over the pairs
that use the slot, bounded here by 2 * 2^-24 * q_slot * S_slot with q_slot and S_slot the
number and absolute sum of the slot's terms."""

import numpy as np
import pytest
from _util import spq, torch_dev

import gen

pytestmark = pytest.mark.gpu


def _graph(kind):
    if kind == "ties":  # weights 1..2: ties everywhere
        g = gen.graphs.grid4(60, 50, wmax=2, seed=3)
        return g, *gen.partition.grid_blocks(60, 50, 13, 11)
    if kind == "holes":  # unreachable pairs, components cut off
        g = gen.graphs.grid_holes(3000, 0.35, wmax=5, seed=4)
        return g, *gen.partition.kdtree(g.xy, 150)
    if kind == "wide":  # more than 256 boundary vertices in a component
        g = gen.graphs.grid4(200, 16, wmax=9, seed=5)
        return g, (np.arange(3200) // 200 % 2).astype(np.int32), 2
    if kind == "single":  # one component: no boundary graph at all
        g = gen.graphs.grid4(30, 20, wmax=9, seed=6)
        return g, np.zeros(600, np.int32), 1
    g = gen.graphs.delaunay(4096, seed=7, weight="f32_lognormal")
    return g, *gen.partition.rcb(g.xy, 4)


@pytest.mark.parametrize("kind", ["ties", "holes", "wide", "single", "float"])
def test_large_batches_take_the_same_walks(kind):
    m = spq()
    torch, dev = torch_dev()
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    g, part, k = _graph(kind)
    q, small, max_len = 12000, 500, 70  # (some rows truncated)
    h = m.spq_build(g.n, T(g.row_ptr), T(g.col), T(g.w), T(part), k)
    rng = np.random.default_rng(1)
    pairs = T(rng.integers(0, g.n, size=(q, 2)).astype(np.int32))
    pairs[7, 1] = pairs[7, 0]
    up = T(rng.normal(size=q).astype(np.float32))
    dist, saved = m.spq_query_saved(h, pairs)
    verts, lens = m.spq_query_paths(h, pairs, saved, max_len)
    gw = torch.zeros(g.col.shape[0], dtype=torch.float32, device=dev)
    m.spq_query_backward(h, pairs, saved, up, gw)
    ref, mag, num = torch.zeros_like(gw), torch.zeros_like(gw), torch.zeros_like(gw)
    for a in range(0, q, small):
        p, s = pairs[a : a + small].contiguous(), saved[a : a + small].contiguous()
        v, n = m.spq_query_paths(h, p, s, max_len)
        assert torch.equal(n, lens[a : a + small])
        there = torch.arange(max_len, device=dev)[None, :] < n[:, None]
        assert torch.equal(v[there], verts[a : a + small][there])
        u = up[a : a + small].contiguous()
        m.spq_query_backward(h, p, s, u, ref)
        m.spq_query_backward(h, p, s, u.abs(), mag)
        m.spq_query_backward(h, p, s, torch.ones_like(u), num)
    m.spq_query_status(h)
    assert int((lens > max_len).sum()) > 0 or kind in ("single", "float", "holes")
    tol = 2.0 * 2.0**-24 * num.double() * mag.double()
    assert bool(((gw - ref).double().abs() <= tol).all())
    h.free()
