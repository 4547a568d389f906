"""The automatic choice of kernel -- many steps per launch for small systems,
the pipelined step beyond, with one species or several -- against the whole-block step kernel (threads = 512), which runs one step per
launch: states, traces, measurements and histograms bit for bit, over every
split of the steps the buffer rotation distinguishes (1, 2, 3, even, odd, more
than one launch), every model and boundary, species, tiles at the edge of the
staging area and spilled records."""
from __future__ import annotations

import numpy as np
import pytest

import paper_2211_15630_gb300 as A
from tests.gpu_helpers import params
from tests.inputs import clustered_state, uniform_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    return A.load()


def pair(species=None, **kw):
    out = []
    for threads in (0, 512):
        p = params(threads=threads, **kw)
        if species:
            A.set_species(p, *species)
        out.append(p)
    return out


def same_state(a, b, n):
    for u, v in zip(A.aap_get_state(a, n), A.aap_get_state(b, n)):
        assert np.array_equal(u, v)


SPECIES = ([700, 1000, 1301], [0.5, 0.3, 0.4], [0.3, 0.5, 0.2], [0.0, 0.1, -0.2],
           [[1.0, 0.5, -0.5], [0.2, 1.0, 3000.0], [0.0, 2.0, 1.0]])
WEAK = SPECIES[:4] + ([[1.0, 0.5, -0.5], [0.2, 1.0, 30.0], [0.0, 2.0, 1.0]],)
CASES = [
    (dict(n=1000, lx=32.0, ly=32.0, eta=0.4, seed=3), None),
    (dict(n=3001, lx=41.3, ly=29.7, eta=0.3, seed=4, bx=1, by=1), None),
    (dict(n=3001, lx=41.3, ly=29.7, eta=0.2, seed=5, model=A.AAP_NVM, by=1), None),
    (dict(n=3001, lx=37.0, ly=33.0, eta=0.4, v=1.0, seed=6, model=A.AAP_LANGEVIN, bx=1), None),
    (dict(n=3001, lx=37.0, ly=33.0, eta=0.4, v=1.0, seed=6, model=A.AAP_LANGEVIN, order=2, weight=A.AAP_H_ONE), None),
    (dict(n=3001, lx=37.0, ly=33.0, seed=7), SPECIES),
    (dict(n=3001, lx=37.0, ly=33.0, seed=8, model=A.AAP_LANGEVIN, bx=1, by=1), SPECIES),
    (dict(n=3001, lx=37.0, ly=33.0, seed=8, model=A.AAP_LANGEVIN, order=3, by=1), WEAK),
    (dict(n=40000, lx=150.0, ly=131.0, eta=0.3, seed=9), None),
    (dict(n=120000, lx=260.0, ly=231.0, eta=0.3, seed=10, model=A.AAP_LANGEVIN, v=1.0), None),
    (dict(n=60000, lx=160.0, ly=171.0, eta=0.3, seed=10, model=A.AAP_LANGEVIN, v=1.0),
     ([20000, 20000, 20000],) + WEAK[1:]),
    (dict(n=60000, lx=160.0, ly=171.0, seed=11, model=A.AAP_LANGEVIN, order=2, weight=A.AAP_H_ONE, bx=1),
     ([30000, 0, 30000],) + SPECIES[1:]),
    (dict(n=60001, lx=160.0, ly=171.0, seed=12, by=1), ([1, 30000, 30000],) + WEAK[1:]),
    (dict(n=60001, lx=160.0, ly=171.0, seed=13, model=A.AAP_NVM), ([20001, 30000, 10000],) + WEAK[1:]),
    (dict(n=7, lx=3.0, ly=3.2, eta=0.3, seed=11), None),
    (dict(n=0, lx=9.0, ly=9.0, eta=0.3, seed=12), None),
]


@pytest.mark.parametrize("kw,species", CASES)
def test_equal_to_one_step_per_launch(kw, species):
    p, q = pair(species, **kw)
    h1, h2 = A.aap_create(p), A.aap_create(q)
    try:
        for steps in (1, 2, 3, 4, 31, 70):
            A.aap_step(h1, steps)
            A.aap_step(h2, steps)
            same_state(h1, h2, p.n)
        assert np.array_equal(A.aap_phi_trace(h1, 37), A.aap_phi_trace(h2, 37))
        for steps in (1, 40):
            A.aap_measure(h1, steps)
            A.aap_measure(h2, steps)
        A.aap_step(h1, 5)
        A.aap_step(h2, 5)
        if p.n:
            r1, r2 = A.aap_get_results(h1), A.aap_get_results(h2)
            assert list(r1.p) == list(r2.p) and list(r1.q) == list(r2.q) and list(r1.nbar) == list(r2.nbar)
            for u, v in zip(A.aap_get_histograms(h1, 100, 100), A.aap_get_histograms(h2, 100, 100)):
                assert np.array_equal(u, v)
            assert np.array_equal(A.aap_step_neighbours(h1, p.n), A.aap_step_neighbours(h2, p.n))
        same_state(h1, h2, p.n)
        o1, o2 = A.aap_observe(h1), A.aap_observe(h2)
        assert (o1.phi, o1.step) == (o2.phi, o2.step) and (p.n == 0 or o1.mean_neighbours == o2.mean_neighbours)
    finally:
        A.aap_destroy(h1)
        A.aap_destroy(h2)


@pytest.mark.parametrize("capacity,w", [(0.0, 6.0), (2.0, 12.0), (0.0, 2.0)])
def test_dense_tiles_and_spilled_records(capacity, w):
    """A dense square: tiles beyond the staging area (global scratch) and, with
    an explicit capacity, regions that overflow into the spill list."""
    n = 9000
    p, q = pair(n=n, lx=40.0, ly=40.0, eta=0.3, seed=21, capacity=capacity)
    c = clustered_state(n // 3, 40.0, 40.0, 5, 13.0, 30.0, w)
    u = uniform_state(n - n // 3, 40.0, 40.0, 6)
    x, y, th = (np.concatenate([a, b]) for a, b in zip(c, u))
    h1, h2 = A.aap_create(p), A.aap_create(q)
    try:
        for h in (h1, h2):
            A.aap_set_state(h, x, y, th.astype(np.float32), 5)
        for steps in (1, 2, 5, 40):
            A.aap_step(h1, steps)
            A.aap_step(h2, steps)
            same_state(h1, h2, n)
    finally:
        A.aap_destroy(h1)
        A.aap_destroy(h2)


def test_withheld_arrival_ends_with_a_status():
    """The grid barrier's wait is bounded: a withheld arrival ends the launch
    with AAP_ETIMEOUT, and the handle works again after aap_set_state."""
    n = 3000
    p, q = pair(n=n, lx=40.0, ly=40.0, eta=0.3, seed=23)
    h1, h2 = A.aap_create(p), A.aap_create(q)
    x, y, th = uniform_state(n, 40.0, 40.0, 8)
    th = th.astype(np.float32)
    try:
        A.aap_test_pipe_wait(20_000_000, 1)
        A.aap_step(h1, 40)
        with pytest.raises(A.AapError) as e:
            A.aap_sync(h1)
        assert e.value.code == A.AAP_ETIMEOUT
        A.aap_test_pipe_wait(0, 0)
        for h in (h1, h2):
            A.aap_set_state(h, x, y, th, 0)
            A.aap_step(h, 50)
        same_state(h1, h2, n)
    finally:
        A.aap_test_pipe_wait(0, 0)
        A.aap_destroy(h1)
        A.aap_destroy(h2)
