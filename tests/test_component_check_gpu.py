"""Component tables stored as int32 by their own back-substitution (needs a GPU).

The float32 tables of an int32 graph are exact below 2^24 and checked: a component in the
elimination form (more than 128 rows, up to 4,096) is stored as integers by its
back-substitution, one in Floyd-Warshall form is converted afterwards.  Paths without edges
between components, so that only the component check can notice: the longest distance is
2^24 - 1 (kept) or 2^24 (rebuilt in int32) in a component of either form, at the edges of the
tile, alone and beside others.  Distances must equal the path's prefix sums exactly.
"""

import numpy as np
import pytest

from _util import spq

pytestmark = pytest.mark.gpu

TWO24 = 1 << 24
ARITH_I32, ARITH_F32 = 1, 2


def _paths(sizes, longest, total):
    """Disjoint paths, one component each; component `longest` has length `total`."""
    rows, cols, ws, part, pos = [], [], [], [], []
    base = 0
    for c, s in enumerate(sizes):
        if s > 1:
            t = total if c == longest else 7 * (s - 1) + 3
            w = np.full(s - 1, t // (s - 1), np.int64)
            w[0] += t - w.sum()
        else:
            w = np.zeros(0, np.int64)
        a = base + np.arange(s - 1)
        rows += [a, a + 1]
        cols += [a + 1, a]
        ws += [w, w]
        part.append(np.full(s, c, np.int32))
        pos.append(np.concatenate([[0], np.cumsum(w)]))
        base += s
    r, c, w = np.concatenate(rows), np.concatenate(cols), np.concatenate(ws)
    o = np.lexsort((c, r))
    rp = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=base))]).astype(np.int64)
    return dict(n=base, row_ptr=rp, col=c[o].astype(np.int32), w=w[o].astype(np.int32), part=np.concatenate(part),
                k=len(sizes)), pos


def _check(h, sizes, pos, arith):
    assert h.stats()["arith"] == arith
    base = 0
    for s, p in zip(sizes, pos):
        v = np.arange(s)
        pairs = (base + np.stack(np.meshgrid(v, v, indexing="ij"), -1).reshape(-1, 2)).astype(np.int32)
        assert np.array_equal(spq().spq_query(h, pairs).reshape(s, s), np.abs(p[:, None] - p[None, :]))
        base += s


SIZES = [(132,), (128,), (1, 129, 60, 257), (300, 125, 2), (140, 128, 260)]


@pytest.mark.parametrize("total,arith", [(TWO24 - 1, ARITH_F32), (TWO24, ARITH_I32)])
@pytest.mark.parametrize("sizes", SIZES)
def test_longest_distance_in_each_component(sizes, total, arith):
    s = spq()
    cases = [(j, *_paths(sizes, j, total)) for j in range(len(sizes)) if sizes[j] > 1]
    for j, g, pos in cases:
        h = s.spq_build(g["n"], g["row_ptr"], g["col"], g["w"], g["part"], g["k"])
        _check(h, sizes, pos, arith)
        s.spq_free(h)


@pytest.mark.parametrize("long_one", [None, 0, 1, 4])
def test_batch(long_one):
    s = spq()
    made = [_paths(z, len(z) - 1, TWO24 if i == long_one else TWO24 - 1) for i, z in enumerate(SIZES)]
    hs = s.spq_build_many([(g["n"], g["row_ptr"], g["col"], g["w"], g["part"], g["k"]) for g, _ in made])
    for h, z, (_, pos) in zip(hs, SIZES, made):
        _check(h, z, pos, ARITH_F32 if long_one is None else ARITH_I32)
    for h in hs:
        s.spq_free(h)
