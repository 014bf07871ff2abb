"""The recorded path walks in every form they have: boundary vertices held in four, six and eight
registers a lane (components of up to 128, 192 and 256 boundary vertices, and more), pairs taken
in the order of their target's component (tables of 64 MB and more, from 16,384 pairs) or in their
own, a graph without boundary vertices, pairs out of range and equal, each against the same pairs
in small batches, which search every hop.  The launch counts show which form ran; the gradients'
tolerance is that of test_walk_records_gpu."""

import numpy as np
import pytest
from _util import spq, torch_dev

import gen

pytestmark = pytest.mark.gpu


def _blocks(side, b, f32=False):
    g = gen.graphs.grid4(side, side, wmax=1000, seed=side)
    if f32:
        g = gen.Graph(g.n, g.row_ptr, g.col, g.w.astype(np.float32), g.xy)
    return g, *gen.partition.grid_blocks(side, side, b, b)


CASES = {  # widest component, whether the pairs are sorted
    "four registers": (lambda: _blocks(96, 32), 124, False),
    "six registers": (lambda: _blocks(120, 40), 156, True),
    "six registers, floats": (lambda: _blocks(120, 40, True), 156, True),
    "eight registers": (lambda: _blocks(165, 55), 216, True),
    "past eight registers": (lambda: _blocks(210, 70), 276, True),
    "no boundary": (lambda: (gen.graphs.grid4(30, 20, wmax=9, seed=6), np.zeros(600, np.int32), 1), 0, False),
}


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("q", [16_000, 20_000])
def test_recorded_walks(name, q):
    m = spq()
    torch, dev = torch_dev()
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    make, max_nb, tables = CASES[name]
    g, part, k = make()
    small, max_len = 500, 600
    h = m.spq_build(g.n, T(g.row_ptr), T(g.col), T(g.w), T(part), k)
    assert int(h.meta()["nb"].max()) == max_nb
    ordered = tables and q >= 16_384
    rng = np.random.default_rng(1)
    pairs = rng.integers(0, g.n, size=(q, 2)).astype(np.int32)
    pairs[7, 1] = pairs[7, 0]
    pairs[8], pairs[q - 1] = (g.n, 3), (5, -2)
    pairs = T(pairs)
    up = T(rng.normal(size=q).astype(np.float32))
    dist, saved = m.spq_query_saved(h, pairs)
    with pytest.raises(m.SpqError):
        m.spq_query_status(h)
    n0 = m.spq_kernel_launches()
    verts, lens = m.spq_query_paths(h, pairs, saved, max_len)
    n1 = m.spq_kernel_launches()
    gw = torch.zeros(g.col.shape[0], dtype=torch.float32, device=dev)
    m.spq_query_backward(h, pairs, saved, up, gw)
    n2 = m.spq_kernel_launches()
    # slots, hops, the walks (backward: boundary graph, ends, flows); sorted: keys and a pass of three
    assert n1 - n0 == 3 + (4 if ordered else 0)
    assert n2 - n1 == 4 + (1 if max_nb else 0) + (4 if ordered else 0)
    assert lens[8] == -1 and lens[q - 1] == -1 and lens[7] == 1
    ref, mag, num = torch.zeros_like(gw), torch.zeros_like(gw), torch.zeros_like(gw)
    for a in range(0, q, small):
        p, s = pairs[a : a + small].contiguous(), saved[a : a + small].contiguous()
        n0 = m.spq_kernel_launches()
        v, n = m.spq_query_paths(h, p, s, max_len)
        assert m.spq_kernel_launches() - n0 == 1
        assert torch.equal(n, lens[a : a + small])
        there = torch.arange(max_len, device=dev)[None, :] < n[:, None]
        assert torch.equal(v[there], verts[a : a + small][there])
        u = up[a : a + small].contiguous()
        m.spq_query_backward(h, p, s, u, ref)
        m.spq_query_backward(h, p, s, u.abs(), mag)
        m.spq_query_backward(h, p, s, torch.ones_like(u), num)
    m.spq_query_status(h)
    tol = 2.0 * 2.0**-24 * num.double() * mag.double()
    assert bool(((gw - ref).double().abs() <= tol).all())
    h.free()
