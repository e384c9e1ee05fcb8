"""Steps on heaps whose blocks hold few objects of the types that the steps
create: with a third type of one 4-byte field and cap_min 32 a block has 10
fish or cars or 8 sharks, fewer than the remainders that a CTA opens a block
for (csrc/dsr_steps.cuh, dsr_create_pending)."""
import numpy as np
import pytest

import oracle as O
from paper_1809_07444_gb300 import apps
from paper_1809_07444_gb300 import workloads as WL
from paper_1809_07444_gb300.heap import Heap, heap_bytes_for_blocks

from helpers import check_invariants, check_stats

pytestmark = pytest.mark.gpu

TUNINGS = [{"cap_min": 32}, {"cap_min": 32, "threads": 64}, {"cap_min": 32, "threads": 1024}]


def _narrow(monkeypatch, types_name):
    types = getattr(apps, types_name) + [[4]]
    monkeypatch.setattr(apps, types_name, types)
    monkeypatch.setattr(apps, "Heap", lambda t, *a, names=None, **kw: Heap(t, *a, **kw))
    return types


def _same(g, o):
    assert g.heap.stats()["error_flags"] == 0
    for a, b in zip(g.dump(), o.dump()):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("tuning", TUNINGS)
@pytest.mark.parametrize("W,H,blocks", [(41, 33, 600), (200, 150, 9000)])  # one cluster (256 threads), and not
def test_wator(monkeypatch, tuning, W, H, blocks):
    types = _narrow(monkeypatch, "WATOR_TYPES")
    k0 = WL.wator_initial(W, H, W)
    kw = dict(fish_breed=2, shark_breed=3)
    g = apps.Wator(W, H, k0, 3, tuning=tuning, heap_bytes=heap_bytes_for_blocks(types, blocks, tuning), **kw)
    assert [g.heap.capacity(t) for t in range(2)] == [10, 8]
    o = O.Wator(W, H, k0, 3, **kw)
    for n in (1, 2, 5, 20):
        c0 = g.heap.counters()
        g.step(n)
        ev = np.sum([o.step(1)[0] for _ in range(n)], axis=0)
        c1 = g.heap.counters()
        assert c1["allocs"] - c0["allocs"] == ev[0] + ev[2]
        _same(g, o)
        check_invariants(g.heap, list(o.counts()) + [0])
    check_stats(g.heap)


@pytest.mark.parametrize("tuning", TUNINGS)
def test_traffic(monkeypatch, tuning):
    types = _narrow(monkeypatch, "TRAFFIC_TYPES")
    R, W = 700, 90
    v0 = WL.traffic_initial(R, W, 5, density=0.2, vmax=5)
    g = apps.Traffic(R, W, v0, 9, alpha=0.9, tuning=tuning, heap_bytes=heap_bytes_for_blocks(types, 9000, tuning))
    assert g.heap.capacity(0) == 10
    o = O.Traffic(R, W, v0, 9, alpha=0.9)
    for n in (1, 2, 5, 20):
        g.step(n)
        o.step(n)
        _same(g, o)
        check_invariants(g.heap, [o.count(), R, 0])
