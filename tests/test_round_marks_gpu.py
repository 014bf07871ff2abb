"""The elimination rounds' tile marks (needs a GPU): which tiles the rounds list follows from the
graph alone, so the same build does the same number of updates every time.  (A round first
turns the marks of the tiles that the last one added into lasting ones, then unmarks the row
tiles that came out all infinite; a tile can be both, so the two passes must not overlap.)"""

import numpy as np
import pytest
from _util import opts, spq, torch_dev

import gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side,leaf,holes", [(60, 40, 0.35), (110, 60, 0.3), (110, 200, 0.0)])
def test_the_same_build_does_the_same_updates(side, leaf, holes):
    m = spq()
    torch, dev = torch_dev()
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    if holes:
        g = gen.graphs.grid_holes(side * side, holes, wmax=100, seed=side)
    else:
        g = gen.graphs.grid4(side, side, wmax=100, seed=side)
    part, k = gen.partition.kdtree(g.xy, leaf)
    args = (g.n, T(g.row_ptr), T(g.col), T(g.w), T(part), k)
    o = opts(bg=m.SPQ_BG_ELIM)
    single, batch = set(), set()
    for _ in range(12):
        h = m.spq_build(*args, opts=o)
        assert 0 < h.stats()["n_bg"] < 4096  # (not autotuned: one form of the rounds)
        single.add(h.stats()["bg_updates"])
        h.free()
        hs = m.spq_build_many([args] * 3, opts=o)
        batch.add(hs[0].stats()["bg_updates"])
        for x in hs:
            x.free()
    assert len(single) == 1 and len(batch) == 1
