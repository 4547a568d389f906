"""More than 16,384 records in one half cell: a ring of particles that move to
its centre without noise or coupling (or a weak one) and meet there on one
step, inside a single call, so that the kernel that runs many steps per launch
is the one that meets them.  Equal bit for bit to the whole-block kernel
(threads = 512), whose ranks inside a cell have the full 16 bits."""
from __future__ import annotations

import numpy as np
import pytest

import paper_2211_15630_gb300 as A
from tests.gpu_helpers import params

pytestmark = pytest.mark.gpu

N, L, RADIUS = 18000, 128.0, 40         # the ring meets after 40 steps of one cell side each


@pytest.fixture(scope="module", autouse=True)
def lib():
    return A.load()


def ring():
    """Aimed at the middle of a half cell inside the tile of 32 x 16 cells at (64, 32)."""
    g = np.random.default_rng(3)
    th = g.permutation(N) * (2.0 * np.pi / N) - np.pi
    return np.mod(80.25 - RADIUS * np.cos(th), L), np.mod(40.5 - RADIUS * np.sin(th), L), th.astype(np.float32)


@pytest.mark.parametrize("gamma,steps", [(0.0, 41), (0.0, 45), (1e-3, 43)])
def test_ring_that_meets_in_one_half_cell(gamma, steps):
    x, y, th = ring()
    out = []
    for threads in (0, 512):
        p = params(n=N, lx=L, ly=L, model=A.AAP_LANGEVIN, v=1.0, dt=1.0, eta=0.0, gamma=gamma, seed=31, threads=threads,
                   tile_w=32, tile_h=16, capacity=40.0)
        h = A.aap_create(p)
        try:
            A.aap_set_state(h, x, y, th, 0)
            A.aap_step(h, steps)
            assert A.aap_test_paths(h)[1] == (0 if threads else steps)
            out.append(A.aap_get_state(h, N) + (A.aap_observe(h).mean_neighbours,))
        finally:
            A.aap_destroy(h)
    if gamma == 0.0:
        # straight paths: on step RADIUS every particle is at the centre, to the
        # fixed-point rounding and the FP32 sine of 45 steps
        d = (steps - RADIUS) * np.array([np.cos(th), np.sin(th)])
        assert np.abs(out[0][0] - (80.25 + d[0])).max() < 1e-3 and np.abs(out[0][1] - (40.5 + d[1])).max() < 1e-3
    for u, v in zip(*out):
        assert np.array_equal(u, v)


@pytest.mark.parametrize("slices", [0, 1, 3])
def test_dense_tiles_share_the_scratch_slices(slices):
    """Eight rings that close in inside one call, in a system of more tiles
    than scratch slices: their tiles outgrow the shared memory at the same time and take
    turns at the slices (with one slice, all of them), some with spilled
    records."""
    m, rings, side, radius = 3000, 8, 512.0, 30
    n = m * rings
    g = np.random.default_rng(9)
    th = np.concatenate([g.permutation(m) * (2.0 * np.pi / m) - np.pi for _ in range(rings)])
    cx = np.repeat([80.25 + 128.0 * (k % 4) for k in range(rings)], m)
    cy = np.repeat([40.5 + 256.0 * (k // 4) for k in range(rings)], m)
    x, y = np.mod(cx - radius * np.cos(th), side), np.mod(cy - radius * np.sin(th), side)
    out = []
    for threads in (0, 512):
        h = A.aap_create(params(n=n, lx=side, ly=side, model=A.AAP_LANGEVIN, v=1.0, dt=1.0, eta=0.0, gamma=1e-3, seed=31,
                                threads=threads, tile_w=32, tile_h=16, capacity=100.0))
        try:
            A.aap_set_state(h, x, y, th.astype(np.float32), 0)
            if not threads and slices:
                A.aap_test_multi_slices(h, slices)
            A.aap_step(h, 36)
            assert A.aap_test_paths(h)[1] == (0 if threads else 36)
            assert A.aap_observe(h).flags & A.AAP_FLAG_SPILLED
            out.append(A.aap_get_state(h, n))
        finally:
            A.aap_destroy(h)
    for u, v in zip(*out):
        assert np.array_equal(u, v)
