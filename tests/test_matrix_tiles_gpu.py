"""Many-to-many distances at the edges of their tiles (64 sources x 128 targets of one
component, 32 boundary vertices a chunk) and small lookups (a CTA per pair), against
spq_query of a large batch (grouped form): integer and float weights, unreachable pairs,
components without and with more than 256 boundary vertices, ids out of range."""

import numpy as np
import pytest
from _util import spq, torch_dev
from test_walk_records_gpu import _graph

pytestmark = pytest.mark.gpu


def _handle(kind):
    m = spq()
    torch, dev = torch_dev()
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    g, part, k = _graph(kind)
    return m, torch, T, g, m.spq_build(g.n, T(g.row_ptr), T(g.col), T(g.w), T(part), k)


def _same(a, b, torch, exact):
    if exact:
        return torch.equal(a.view(torch.int32), b.view(torch.int32))
    # (float weights: the matrix sums from the source's side, spq_query from the lower
    #  component's: three-term sums of at most 200 hops, each rounding 2^-24 relative)
    return bool((((a - b).abs() <= 1.2e-5 * b.abs()) | (a == b) | (a.isnan() & b.isnan())).all())


@pytest.mark.parametrize("kind", ["ties", "holes", "wide", "single", "float"])
@pytest.mark.parametrize("ns,nt", [(1, 1), (63, 127), (64, 128), (65, 129), (130, 600)])
def test_matrix_tile_edges(kind, ns, nt):
    m, torch, T, g, h = _handle(kind)
    rng = np.random.default_rng(ns)
    src = rng.integers(0, g.n, size=ns).astype(np.int32)
    tgt = (rng.integers(0, g.n) + np.arange(nt)).astype(np.int32) % g.n  # whole runs of a component
    tgt[-1] = src[0]
    if nt > 500:
        src[7], tgt[9] = -1, g.n
    D = m.spq_query_matrix(h, T(src), T(tgt))
    pairs = np.stack(np.meshgrid(src, tgt, indexing="ij"), -1).reshape(-1, 2).astype(np.int32)
    pad = np.zeros((max(0, 4097 - len(pairs)), 2), np.int32)
    ref = m.spq_query(h, T(np.concatenate([pairs, pad])))[: len(pairs)].reshape(ns, nt)
    assert _same(D, ref, torch, kind != "float")
    if nt > 500:
        with pytest.raises(m.SpqError):
            m.spq_query_status(h)
    h.free()


@pytest.mark.parametrize("kind", ["ties", "holes", "wide", "single", "float"])
@pytest.mark.parametrize("q", [1, 9, 4095])
def test_small_batches_equal_large_ones(kind, q):
    m, torch, T, g, h = _handle(kind)
    rng = np.random.default_rng(q)
    pairs = rng.integers(0, g.n, size=(5000, 2)).astype(np.int32)
    pairs[0] = pairs[0, 0]
    pairs[8] = (3, -5)
    ref = m.spq_query(h, T(pairs))
    got = m.spq_query(h, T(pairs[:q]))
    assert _same(got, ref[:q], torch, True)
    h.free()
