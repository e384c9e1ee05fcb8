"""Steps of the applications over heaps whose types have subtypes
(dsr_heap_set_bases): every do-all of a step visits the subtypes' objects as
well, so a state of which half the objects are of a subtype with its base's
fields advances as the oracle's does."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1809_07444_gb300 import _lib as L
from paper_1809_07444_gb300 import apps
from paper_1809_07444_gb300 import workloads as WL
from paper_1809_07444_gb300.heap import Heap

from helpers import check_invariants

pytestmark = pytest.mark.gpu


def _with_subtypes(monkeypatch, types_name, make):
    """make() on a heap of the application's types and a subtype of each;
    the objects of each type whose first field is even are then replaced by
    copies of the subtype. Returns the application and {old handle: new handle}."""
    types = getattr(apps, types_name)
    n = len(types)
    monkeypatch.setattr(apps, types_name, types + types)
    monkeypatch.setattr(apps, "Heap", lambda t, *a, names=None, **kw: Heap(t, *a, **kw))
    g = make()
    moved = {}
    for t in range(n):
        f, h = g.heap.dump(t)
        if not len(h):
            continue
        g.heap.parallel_do(t, L.METHOD_CLONE, L.CloneArgs(n + t, 0))
        g.heap.parallel_do(n + t, L.METHOD_DELETE_IF, L.DeleteIfArgs(2, 1))
        g.heap.parallel_do(t, L.METHOD_DELETE_IF, L.DeleteIfArgs(2, 0))
        f2, h2 = g.heap.dump(n + t)
        new = {tuple(r): int(k) for r, k in zip(f2, h2)}
        moved[t] = {int(k): new[tuple(r)] for r, k in zip(f, h) if tuple(r) in new}
        assert 0 < len(moved[t]) == len(h2)
    dump = g.heap.dump

    def both(t):
        f, h = dump(t)
        f2, h2 = dump(n + t)
        return np.concatenate([f, f2]), np.concatenate([h, h2])

    g.heap.dump = both
    g.heap.set_bases([-1] * n + list(range(n)))
    return g, moved


def _remap(ws, at, dtype, count, fn):
    """Apply fn to the table of `count` dtype words at byte `at` of a workspace."""
    size = np.dtype(dtype).itemsize * count
    words = ws[at: at + size].cpu().numpy().view(dtype)
    ws[at: at + size].copy_(torch.from_numpy(fn(words).view(np.uint8)))


def _same(g, o, step):
    for a, b in zip(g.dump(), o.dump()):
        assert np.array_equal(a, b), step
    assert g.heap.stats()["error_flags"] == 0
    check_invariants(g.heap)


SIZES = [(41, 33), (150, 131)]  # steps in one cluster, and kernel by kernel


@pytest.mark.parametrize("size", SIZES)
def test_life(monkeypatch, size):
    W, H = size
    s0 = WL.gol_initial(W, H, W)
    g, moved = _with_subtypes(monkeypatch, "GOL_TYPES", lambda: apps.Gol(W, H, s0))
    _remap(g.workspace, 0, np.uint64, W * H,
           lambda w: np.array([moved[0].get(int(r), int(r)) for r in w], dtype=np.uint64))
    o = O.Gol(W, H, s0)
    for n in (1, 2, 5):
        g.step(n)
        o.step(n)
        _same(g, o, n)


@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("timed", [False, True])
def test_wator(monkeypatch, size, timed):
    W, H = size
    k0 = WL.wator_initial(W, H, W)
    g, moved = _with_subtypes(monkeypatch, "WATOR_TYPES", lambda: apps.Wator(W, H, k0, 3))
    both = {**moved[0], **moved[1]}
    _remap(g.workspace, 0, np.uint32, W * H,
           lambda w: np.array([(both.get(int(r) >> 2, int(r) >> 2) << 2) | (int(r) & 3) if r else 0 for r in w],
                              dtype=np.uint32))  # 0: an empty cell
    o = O.Wator(W, H, k0, 3)
    if timed:
        g.phase_timing(100)
    for n in (1, 2, 20):
        c0, visits = g.heap.counters(), 0
        for _ in range(n):
            fish, sharks = o.counts()
            starved = o.step(1)[0][3]
            visits += 2 * fish + sharks + 2 * (sharks - starved)
        g.step(n)
        assert g.heap.counters()["visits"] - c0["visits"] == visits
        _same(g, o, n)


@pytest.mark.parametrize("periodic", [False, True])
def test_traffic(monkeypatch, periodic):
    R, L_ = 101, 203
    v0 = WL.traffic_initial(R, L_, 5, density=0.2, vmax=5)
    kw = dict(vmax=5, p=0.25, alpha=0.5, periodic=periodic)
    g, _ = _with_subtypes(monkeypatch, "TRAFFIC_TYPES", lambda: apps.Traffic(R, L_, v0, 9, **kw))
    o = O.Traffic(R, L_, v0, 9, **kw)
    for n in (1, 2, 20):
        g.step(n)
        o.step(n)
        _same(g, o, n)


def test_sugarscape(monkeypatch):
    W, H = 120, 97
    cap, a0 = WL.sugarscape_initial(W, H, 4)
    g, _ = _with_subtypes(monkeypatch, "SUGAR_TYPES", lambda: apps.Sugarscape(W, H, cap, a0, 6))
    o = O.Sugarscape(W, H, cap, a0, 6)
    for n in (1, 2, 40):
        g.step(n)
        o.step(n)
        _same(g, o, n)
