"""What a batch's handles and a query plan hold of the device's memory (needs a GPU)."""

import ctypes

import numpy as np
import pytest
from _util import opts, spq, torch_dev

import gen

pytestmark = pytest.mark.gpu


def _used():
    m = spq()
    torch, _ = torch_dev()
    torch.cuda.synchronize()
    used, reserved = ctypes.c_ulonglong(), ctypes.c_ulonglong()
    assert m._lib.load().spq_pool_usage(0, ctypes.byref(used), ctypes.byref(reserved)) == 0
    return used.value


def _graphs(sizes):
    torch, dev = torch_dev()
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    out = []
    for side, leaf in sizes:
        g = gen.graphs.grid4(side, side, wmax=100, seed=side)
        part, k = gen.partition.kdtree(g.xy, leaf)
        out.append((g.n, T(g.row_ptr), T(g.col), T(g.w), T(part), k))
    return out


@pytest.mark.parametrize("bg", [0, 1])
def test_handles_hold_their_footprints(bg):
    """Boundary graphs of 6,700 to 16,800 slots, in aligned pieces (0) or packed (1): the pieces'
    padding is held as far as the order uses it, and counted."""
    m = spq()
    gs = _graphs([(40, 60), (150, 24), (230, 24)])
    before = _used()
    hs = m.spq_build_many(gs, opts=opts(bg=bg))
    held = _used() - before
    told = sum(h.stats()["footprint_bytes"] for h in hs)
    assert told <= held <= told + (8 << 20)  # (the pool hands out whole units)
    for h in hs:
        h.free()
    assert _used() == before


@pytest.mark.parametrize("q", [50_000, 3_000_000])
def test_a_query_plan_holds_bounded_scratch(q):
    """Four instances in flight take four scratches (about 90 bytes a pair of the largest
    instance), together at most 256 MiB; a larger instance takes one, as it needs anyway."""
    m = spq()
    torch, dev = torch_dev()
    hs = m.spq_build_many(_graphs([(40, 60)] * 4))
    pairs = [torch.randint(0, 1600, (q, 2), dtype=torch.int32, device=dev) for _ in hs]
    ref = [m.spq_query(h, p) for h, p in zip(hs, pairs)]
    before = _used()
    plan = m.spq_query_plan(hs, pairs)
    assert _used() - before <= max(256 << 20, 96 * q) + (8 << 20)
    for out, r in zip(plan.run(), ref):
        assert torch.equal(out, r)
    plan.free()
    assert _used() == before
    for h in hs:
        h.free()
