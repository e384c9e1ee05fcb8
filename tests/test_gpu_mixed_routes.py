"""Steps of one heap by different routes in turn: a small wa-tor heap takes its
untimed steps in one cluster launch and its timed ones kernel by kernel
(csrc/dsr_wator.cu), and either must find the block lists empty whatever the
steps before it left, also after a checkpoint."""
import numpy as np
import pytest

import oracle as O
from paper_1809_07444_gb300 import workloads as WL
from paper_1809_07444_gb300.apps import Wator

from helpers import check_invariants

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("timed", [1, 2, 3])
@pytest.mark.parametrize("resume", [False, True])
def test_wator_untimed_steps_after_timed_ones(timed, resume):
    W, H = 64, 49
    k0 = WL.wator_initial(W, H, timed)
    g, o = Wator(W, H, k0, 5), O.Wator(W, H, k0, 5)

    def both(n):
        c0 = g.heap.counters()
        g.step(n)
        ev = np.sum([o.step(1)[0] for _ in range(n)], axis=0)
        c1 = g.heap.counters()
        assert c1["allocs"] - c0["allocs"] == ev[0] + ev[2]
        assert c1["frees"] - c0["frees"] == ev[1] + ev[3]
        assert g.hash() == o.hash()

    for untimed in (4, 1, 3):
        g.phase_timing(timed)
        both(timed)
        assert g.phase_times()[2] == timed
        if resume:
            g = Wator.restore(g.checkpoint())
        else:
            g.phase_timing(0)
        both(untimed)
    for a, b in zip(g.dump(), o.dump()):
        assert np.array_equal(a, b)
    check_invariants(g.heap, list(o.counts()))
