"""Heaps with little room: a do-all that frees memory runs before one that
needs it, as its order in the step says."""
import numpy as np
import pytest

import oracle as O
from paper_1809_07444_gb300.apps import GOL_TYPES, Gol, GolBatch
from paper_1809_07444_gb300.heap import heap_bytes_for_blocks

from helpers import check_invariants

pytestmark = pytest.mark.gpu


def _blinkers(nx, ny):
    """nx x ny blinkers, each in 5 x 5 cells of its own: every generation two of three cells die and two are born."""
    s = np.zeros((5 * ny, 5 * nx), dtype=np.uint8)
    s[2::5, 1::5] = s[2::5, 2::5] = s[2::5, 3::5] = 1
    return s


# 32 x 20 blinkers: 1920 alive in 30 blocks at least, 1280 born a generation,
# 20 blocks' worth; the heap has 12 blocks of room. One cluster, and kernel by kernel.
@pytest.mark.parametrize("tuning", [None, {"threads": 128}])
@pytest.mark.parametrize("batch", [False, True])
def test_life_with_room_for_the_births_only_after_the_deaths(tuning, batch):
    s0 = _blinkers(32, 20)
    H, W = s0.shape
    blocks = -(-W * H // 42) + 30 + 12
    o = O.Gol(W, H, s0)
    if batch:
        b = GolBatch(64 << 20, max_instances=2, tuning=tuning)
        slot = b.add(W, H, s0, n_blocks=blocks)
        heap, step, hashes = b.heap(slot), b.step, lambda: b.hash(slot)
    else:
        g = Gol(W, H, s0, heap_bytes=heap_bytes_for_blocks(GOL_TYPES, blocks, tuning), tuning=tuning)
        heap, step, hashes = g.heap, g.step, g.hash
    assert heap.layout().n_blocks == blocks and heap.stats()["error_flags"] == 0
    for n in (1, 2, 7):
        step(n)
        o.step(n)
        assert heap.stats()["error_flags"] == 0
        assert hashes() == o.hash()
    check_invariants(heap, [W * H, o.alive_count()])


def test_traffic_sources_find_room_beside_the_cars():
    # 1838 cars in 29 blocks and 100 sources in two at least: 34 blocks, of
    # which partly filled blocks of cars may take three more
    from paper_1809_07444_gb300 import workloads as WL
    from paper_1809_07444_gb300.apps import TRAFFIC_TYPES, Traffic

    R, L = 100, 90
    v0 = WL.traffic_initial(R, L, 5, density=0.2, vmax=5)
    assert (v0 >= 0).sum() == 1838
    for _ in range(5):
        g, o = (f(R, L, v0, 9, **kw) for f, kw in (
            (Traffic, {"heap_bytes": heap_bytes_for_blocks(TRAFFIC_TYPES, 34)}), (O.Traffic, {})))
        for n in (0, 20):
            g.step(n)
            if n:
                o.step(n)
            assert g.heap.stats()["error_flags"] == 0
            for a, b in zip(g.dump(), o.dump()):
                assert np.array_equal(a, b)
