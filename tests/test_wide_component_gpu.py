"""A component with more than 46,340 boundary vertices (needs a GPU): the flows of its clique
edges are |B|^2 > 2^31 cells, so a cell's place in the component's table needs 64 bits.

47,000 vertices, all of them on the boundary of one component: leaves, each on one of 216 middle
vertices, those on the top one.  The only light edge out leads from the top vertex to a hub in
the other component; every other vertex has a heavy one (which makes it a boundary vertex).
The path from a leaf to the hub is leaf - middle - top - hub, of ascending numbers, so the
recorded walk takes the clique edges (leaf, middle) and (middle, top): for leaves from 45,691 on
the first lies past cell 2^31.  Gradients are path counts: exact."""

import numpy as np
import pytest
from _util import graph_from_edges, spq, torch_dev

pytestmark = pytest.mark.gpu


def test_flows_past_2_31_cells():
    m = spq()
    torch, dev = torch_dev()
    n0, mid, hubs = 47_000, 216, 47
    n = n0 + hubs
    leaf, top = np.arange(n0 - 1 - mid), n0 - 1
    middle = n0 - 1 - mid + np.arange(mid)
    above = middle[leaf % mid]
    edges = [(a, b, 1 + a % 7) for a, b in zip(leaf.tolist(), above.tolist())]
    edges += [(a, top, 3) for a in middle.tolist()]
    edges += [(a, n0 + a // 1000, 10_000) for a in range(n0 - 1)] + [(top, n0, 2)]
    g = graph_from_edges(n, edges)
    part = (np.arange(n) >= n0).astype(np.int32)
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    h = m.spq_build(n, T(g.row_ptr), T(g.col), T(g.w), T(part), 2)
    assert h.meta()["nb"][0] == n0

    first = -(-(2**31) // n0)  # leaf * n0 >= 2^31 from here on
    start = np.arange(first, leaf[-1] + 1)
    times = 520  # 21 q sqrt(n) > sum |C||B(C)|: the recorded walks
    pairs = np.stack([start, np.full_like(start, n0)], 1).astype(np.int32)
    assert 21.0 * times * len(start) * np.sqrt(n) > 7.5e6 + n0 * n0 + hubs * hubs
    dist, saved = m.spq_query_saved(h, T(pairs))
    assert np.array_equal(dist.cpu().numpy(), 1 + start % 7 + 3 + 2)
    assert np.array_equal(saved.cpu().numpy(), np.stack([start, np.zeros_like(start)], 1))
    gw = torch.zeros(g.col.shape[0], dtype=torch.float32, device=dev)
    m.spq_query_backward(h, T(pairs).repeat(times, 1), saved.repeat(times, 1),
                         torch.ones(times * len(start), dtype=torch.float32, device=dev), gw)
    torch.cuda.synchronize()
    m.spq_query_status(h)
    h.free()

    ref = np.zeros(g.col.shape[0], np.float32)
    slot = {}

    def add(a, b, x):
        if (a, b) not in slot:
            row = g.col[g.row_ptr[a] : g.row_ptr[a + 1]]
            slot[a, b] = g.row_ptr[a] + int(np.nonzero(row == b)[0][0])
        ref[slot[a, b]] += x

    for a in start.tolist():
        add(a, int(above[a]), times)
        add(int(above[a]), top, times)
        add(top, n0, times)
    assert np.array_equal(gw.cpu().numpy(), ref)
