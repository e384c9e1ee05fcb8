"""FP32 pair forces where the cube of the distance leaves FP32's normal range
but the mass over it does not: distances of 1e13 to 1e16 between large masses,
and softening lengths whose inverse cube overflows. One step against the FP64
oracle at the bar of the other n-body tests (1e-4 relative; at rest before)."""
import os

import numpy as np
import pytest

import oracle as O
from paper_1809_07444_gb300.apps import NBody

from test_gpu_nbody import _compare

pytestmark = pytest.mark.gpu


def _one_step(rows, pairs, **kw):
    rows = rows.astype(np.float32).astype(np.float64)
    g = NBody(rows, pairs=pairs, r_near=0.0, **kw)
    O.set_threads(os.cpu_count() or 8)
    o = O.NBody(rows, **kw)
    g.step(1)
    o.step(1)
    _compare(g.dump(), o.dump())
    assert g.heap.stats()["error_flags"] == 0


def _far(n, scale, mass, rng):
    rows = np.zeros((n, 7))
    rows[:, :3] = scale * rng.uniform(-1, 1, (n, 3))
    rows[:, 6] = mass * rng.uniform(0.1, 1, n)
    return rows


@pytest.mark.parametrize("pairs", ["fp32", "fp64"])
@pytest.mark.parametrize("scale", [1e11, 3e12, 1e13, 1e14, 1e16])
def test_large_masses_far_apart(scale, pairs):
    # G sets the velocities of one step to about 1; a mass over eps^3 is within
    # FP32's range, as the term of a body on itself needs it to be
    rows = _far(300, scale, 1e30, np.random.default_rng(1))
    _one_step(rows, pairs, G=scale ** 2 / 1e30 / 100, dt=1.0, eps=1e6, r_merge=1e-9)


def test_far_bodies_among_many_near_ones():
    # tiles of both kinds in the form for many bodies
    rng = np.random.default_rng(2)
    rows = np.zeros((16500, 7))
    rows[:, :3] = rng.random((16500, 3))
    rows[:, 6] = 10 ** rng.uniform(-3, 0, 16500)
    rows[:64] = _far(64, 1e14, 1e27, rng)
    _one_step(rows, "fp32", G=1.0, dt=1e-4, eps=1e-3, r_merge=1e-9)


@pytest.mark.parametrize("eps", [1e-12, 1e-13, 1e-14, 2e-16])
def test_small_softening_and_masses(eps):
    rng = np.random.default_rng(3)
    rows = np.zeros((300, 7))
    rows[:, :3] = rng.random((300, 3))
    rows[:, 6] = 1e-12 * rng.uniform(0.1, 1, 300)
    _one_step(rows, "fp32", G=1e12, dt=1e-4, eps=eps, r_merge=1e-9)
