"""Initial states placed by whole CTAs (csrc/dsr_bulk.cuh): sizes around a
chunk and a block, other block capacities and fan-outs, a heap with exactly
as many slots as objects, and slow paths that are made to fail."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TUNINGS = [None, {"cap_min": 32}, {"fanout": 16}]


@pytest.mark.parametrize("shape", [(3, 3), (3, 85), (16, 16), (3, 86), (63, 65), (64, 64), (37, 111), (701, 997),
                                   (2048, 1025)])
@pytest.mark.parametrize("tuning", TUNINGS)
def test_gol_cells_and_alive(shape, tuning):
    from paper_1809_07444_gb300 import workloads as WL
    from paper_1809_07444_gb300.apps import Gol

    from helpers import check_stats

    W, H = shape
    start = WL.gol_initial(W, H, seed=W * 1000 + H)
    g = Gol(W, H, start, tuning=tuning)
    cells, alive = g.dump()
    idx = np.arange(W * H)
    assert np.array_equal(cells, np.stack([start.reshape(-1), np.zeros_like(idx), idx], 1))
    on = np.flatnonzero(start.reshape(-1))
    expect = np.stack([on % W, on // W], 1)
    assert np.array_equal(alive, expect[np.lexsort(expect.T[::-1])])
    st = check_stats(g.heap)
    assert st["error_flags"] == 0
    c = g.heap.counters()
    assert c["allocs"] == W * H + len(on) and c["new_blocks"] == sum(st["allocated_blocks"])


@pytest.mark.parametrize("n", [65, 128, 4096, 4097, 64 * 777])  # two blocks: the smallest heap of this type
def test_heap_with_exactly_enough_slots(n):
    from paper_1809_07444_gb300.apps import NBODY_TYPES, NBody
    from paper_1809_07444_gb300.heap import heap_bytes_for_blocks

    from helpers import check_stats

    rows = np.random.default_rng(n).random((n, 7)).astype(np.float32)
    nb = NBody(rows, heap_bytes=heap_bytes_for_blocks(NBODY_TYPES, -(-n // 64)))
    st = check_stats(nb.heap)
    assert st["live_objects"] == [n] and st["error_flags"] == 0
    d = nb.dump()
    assert np.array_equal(d[:, 0], np.arange(n))
    assert np.array_equal(d[:, 1:].astype(np.float32), rows)


def test_injected_failures_reach_the_bulk_path():
    import ctypes as C

    import torch

    from paper_1809_07444_gb300 import _lib as L
    from paper_1809_07444_gb300.apps import NBODY_TYPES, NBody
    from paper_1809_07444_gb300.heap import _stream_ptr

    from helpers import check_stats

    n = 4096
    nb = NBody(np.random.default_rng(1).random((n, 7)).astype(np.float32))
    assert nb.heap.types == NBODY_TYPES
    L.check(nb.lib.dsr_nbody_destroy(nb.handle))
    nb.handle = None
    nb.heap.reset()
    nb.heap.inject_oom(1 << 30)
    h = C.c_void_p()
    L.check(nb.lib.dsr_nbody_create(nb.heap.handle, C.byref(nb.params), C.c_void_p(nb._rows.data_ptr()), n,
                                    C.c_void_p(nb.workspace.data_ptr()), nb.log_cap, _stream_ptr(), C.byref(h)))
    nb.handle = h
    torch.cuda.synchronize()
    st = check_stats(nb.heap)
    assert st["live_objects"] == [0] and st["error_flags"] == L.ERR_OOM
