"""The back-substitution's work order by levels, whole tiles and column strips: the
boundary matrix by elimination equals the one by Floyd-Warshall, entry for entry, where
every level is split into strips (few tiles), where only the narrow levels are, where row
blocks have no frontier (disconnected boundary graphs), and over several panel launches."""

import numpy as np
import pytest

import gen
import paper_1503_07192_gb300 as spq

pytestmark = pytest.mark.gpu


def _opts(bg, arith, panel):
    o = spq.spq_opts_default()
    o.bg_method, o.comp_method, o.arith, o.bg_panel_mib = bg, bg, arith, panel
    return o


@pytest.mark.parametrize("arith", [spq.SPQ_ARITH_F32, spq.SPQ_ARITH_I32])
@pytest.mark.parametrize("kind,side,leaf,panel", [
    ("grid", 20, 100, 0),      # one or two row blocks: nothing but strips
    ("grid", 64, 256, 0),      # a few row blocks
    ("holes", 150, 200, 0),    # pockets: rows without a frontier
    ("grid", 220, 150, 0),     # levels of both kinds
    ("grid", 220, 150, 1),     # the same in several launches
])
def test_elimination_equals_floyd_warshall(kind, side, leaf, panel, arith):
    if kind == "holes":
        g = gen.graphs.grid_holes(side * side, 0.35, wmax=100, seed=side)
    else:
        g = gen.graphs.grid4(side, side, wmax=100, seed=side)
    part, k = gen.partition.kdtree(g.xy, leaf)
    a = spq.spq_build(g.n, g.row_ptr, g.col, g.w, part, k, _opts(spq.SPQ_BG_ELIM, arith, panel))
    b = spq.spq_build(g.n, g.row_ptr, g.col, g.w, part, k, _opts(spq.SPQ_BG_FW, arith, panel))
    assert np.array_equal(a.bg(), b.bg())
    for c in range(0, k, max(1, k // 5)):
        assert np.array_equal(a.apsp(c), b.apsp(c))
    a.free()
    b.free()


def test_batched_pieces_equal_floyd_warshall():
    """Batched instances whose boundary graphs are ordered in aligned pieces (from 4,096 slots,
    2 to 8 leaf runs side by side), beside smaller ones and one with pockets, against
    Floyd-Warshall of each alone."""
    graphs = []
    for side, leaf, holes in [(40, 60, 0.0), (150, 24, 0.0), (230, 24, 0.0), (170, 20, 0.25)]:
        if holes:
            g = gen.graphs.grid_holes(side * side, holes, wmax=100, seed=side)
        else:
            g = gen.graphs.grid4(side, side, wmax=100, seed=side)
        graphs.append((g, *gen.partition.kdtree(g.xy, leaf)))
    hs = spq.spq_build_many([(g.n, g.row_ptr, g.col, g.w, part, k) for g, part, k in graphs])
    assert max(h.stats()["n_bg"] for h in hs) >= 16384
    for h, (g, part, k) in zip(hs, graphs):
        b = spq.spq_build(g.n, g.row_ptr, g.col, g.w, part, k, _opts(spq.SPQ_BG_FW, spq.SPQ_ARITH_F32, 0))
        assert np.array_equal(h.bg(), b.bg())
        b.free()
    for h in hs:
        h.free()
