"""FP32 pair forces where the cube of the distance leaves FP32's normal range
but the mass over it does not: distances of 1e13 to 1e16 between large masses,
and softening lengths whose inverse cube overflows. One step against the FP64
oracle at the bar of the other n-body tests (1e-4 relative; at rest before).
And FP64 pair forces over that range, to the last bits a state keeps."""
import os

import numpy as np
import pytest

import oracle as O
from paper_1809_07444_gb300.apps import NBODY_TYPES, NBody
from paper_1809_07444_gb300.heap import heap_bytes_for_blocks

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


def test_fp64_terms_to_the_last_bits():
    # One body pulls another: v = G m d (d^2 + eps^2)^-3/2 dt, of the order of
    # one. The state holds v as two FP32 numbers, 2^-48 of it apart at most;
    # the few FP64 roundings before are well below. A wrong coefficient of the
    # series for r^-3 shows far above 2^-44.
    rng = np.random.default_rng(5)
    for r in 10 ** rng.uniform(-15, 15, 60):
        rows = np.zeros((2, 7), dtype=np.float32)
        rows[1, :3] = r * rng.uniform(-1, 1, 3)
        rows[:, 6] = rng.uniform(0.5, 2, 2)
        eps = float(r * rng.uniform(0.01, 1))
        G = float(r * r)
        g = NBody(rows, G=G, eps=eps, dt=1.0, r_merge=0.0, r_near=0.0, pairs="fp64", log_cap=16,
                  heap_bytes=heap_bytes_for_blocks(NBODY_TYPES, 64))
        g.step(1)
        x = rows.astype(np.longdouble)
        d = x[1, :3] - x[0, :3]
        e2 = np.longdouble(eps * eps)
        w = (d @ d + e2) ** np.longdouble(-1.5)
        want = np.stack([d * w * x[1, 6], -d * w * x[0, 6]]) * np.longdouble(G)
        got = g.dump()[:, 4:7]
        assert (abs(got - want) <= 2.0 ** -44 * abs(want)).all(), (r, eps)
