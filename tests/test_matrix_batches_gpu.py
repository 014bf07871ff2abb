"""Many-to-many distances of more sources than one batch of t holds, and of many sources to few
targets (t has columns for the components with targets only), against spq_query of the same
pairs: integer and float weights, unreachable pairs, ids out of range."""

import numpy as np
import pytest
from _util import spq
from test_matrix_tiles_gpu import _handle, _same

pytestmark = pytest.mark.gpu

T_ELEMS = 1 << 24  # most values of t at a time


@pytest.mark.parametrize("kind", ["ties", "holes", "float"])
@pytest.mark.parametrize("nt,batches", [(1, 1), (3, 1), (300, 2)])
def test_many_sources(kind, nt, batches):
    m, torch, T, g, h = _handle(kind)
    rng = np.random.default_rng(nt)
    nb = h.meta()["nb"]  # columns of t with targets everywhere
    ldt = min(h.stats()["n_bg"] + 3 * len(nb), len(nb) * -(-int(nb.max()) // 4) * 4)
    ns = T_ELEMS // ldt + 70 if batches > 1 else 5000
    src = rng.integers(0, g.n, size=ns).astype(np.int32)
    tgt = rng.integers(0, g.n, size=nt).astype(np.int32)
    tgt[0] = src[-1]
    if nt > 1:
        src[ns // 2], src[-2], tgt[1] = -1, g.n, g.n + 5
    if batches > 1:  # (every component has targets)
        part = h.meta()["comp"]
        assert len(np.unique(part[tgt[(tgt >= 0) & (tgt < g.n)]])) > 0.8 * len(nb)
    D = m.spq_query_matrix(h, T(src), T(tgt))
    for a in range(0, ns, 8192):
        s = src[a : a + 8192]
        pairs = np.stack(np.meshgrid(s, tgt, indexing="ij"), -1).reshape(-1, 2).astype(np.int32)
        ref = m.spq_query(h, T(pairs)).reshape(len(s), nt)
        assert _same(D[a : a + 8192], ref, torch, kind != "float")
    if nt > 1:
        with pytest.raises(m.SpqError):
            m.spq_query_status(h)
    h.free()
