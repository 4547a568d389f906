"""Which kernel ran: the equalities of the other tests hold whatever the
automatic choice picks, so the choice itself is pinned here (aap_test_paths,
aap_sur_test_paths)."""
from __future__ import annotations

import numpy as np
import pytest

import paper_2211_15630_gb300 as A
from tests.gpu_helpers import params
from tests.inputs import clustered_state, uniform_state
from tests.test_gpu_multi import CASES, pair

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def lib():
    return A.load()


@pytest.mark.parametrize("kw,species", CASES)
def test_small_systems_run_many_steps_per_launch(kw, species):
    p, q = pair(species, **kw)
    for prm, steps in ((p, 71), (q, 0)):
        h = A.aap_create(prm)
        try:
            A.aap_step(h, 1)
            A.aap_step(h, 70)
            launches, in_them = A.aap_test_paths(h)[:2]
            assert in_them == steps and launches == (4 if steps else 0)      # 1, 31, 32, 7 steps
        finally:
            A.aap_destroy(h)


@pytest.mark.parametrize("calls,launches", [((31, 66), 4), ((30, 5, 32), 3), ((29, 40), 3), ((1, 2, 3, 4), 4), ((67,), 2)])
def test_the_load_is_looked_at_every_32_to_35_steps(calls, launches):
    """Launches end at least every 35 steps counted across calls (31 | 4, 32,
    30; 30 | 5 | 32; 29 | 6, 34; the calls themselves; 32, 35)."""
    h = A.aap_create(params(n=1000, lx=32.0, ly=32.0, eta=0.4, seed=3))
    try:
        for k in calls:
            A.aap_step(h, k)
        assert list(A.aap_test_paths(h)[:2]) == [launches, sum(calls)]
    finally:
        A.aap_destroy(h)


def test_dense_states_leave_many_steps_and_return():
    """A dense spot (inside one tile of 30 x 15 cells) goes to single steps at once; when it has spread (straight
    paths, no coupling) the handle returns to many steps per launch."""
    n, side = 3500, 60.0
    g = np.random.default_rng(5)
    th = g.uniform(-np.pi, np.pi, n).astype(np.float32)
    r = g.uniform(0.0, 0.4, n)
    h = A.aap_create(params(n=n, lx=side, ly=side, model=A.AAP_LANGEVIN, v=1.0, dt=0.5, eta=0.0, gamma=0.0, seed=6))
    try:
        A.aap_set_state(h, 20.2 + r * np.cos(th), 22.2 + r * np.sin(th), th, 0)
        A.aap_step(h, 2)
        assert A.aap_test_paths(h)[0] == 0
        for _ in range(8):
            A.aap_step(h, 32)
            A.aap_sync(h)
        assert A.aap_test_paths(h)[0] > 0
        x, y, t = uniform_state(n, side, side, 7)
        A.aap_set_state(h, x, y, t.astype(np.float32), 0)
        before = A.aap_test_paths(h)[1]
        A.aap_step(h, 10)
        assert A.aap_test_paths(h)[1] == before + 10
    finally:
        A.aap_destroy(h)


def test_spilled_records_count_as_load():
    """An explicit capacity that keeps some 2,000 records of a dense spot in
    the spill list: the regions alone look light (a load of 3,700), the tile is not
    (15,000 with the spilled ones)."""
    n, side = 9000, 60.0
    c = clustered_state(3000, side, side, 5, 20.2, 22.2, 0.8)
    u = uniform_state(n - 3000, side, side, 6)
    x, y, th = (np.concatenate(v) for v in zip(c, u))
    out = []
    for threads in (0, 512):
        h = A.aap_create(params(n=n, lx=side, ly=side, eta=0.3, v=0.1, seed=8, capacity=2.0, threads=threads))
        try:
            A.aap_set_state(h, x, y, th.astype(np.float32), 0)
            A.aap_step(h, 3)
            assert A.aap_test_paths(h)[0] == 0
            assert A.aap_observe(h).flags & A.AAP_FLAG_SPILLED
            out.append(A.aap_get_state(h, n))
        finally:
            A.aap_destroy(h)
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def test_a_windows_first_sample_is_the_observed_state():
    """p and q of a window of one step are those aap_observe gives, bit for
    bit (the window starts on the device, the observation ends on the host)."""
    h = A.aap_create(params(n=1000, lx=32.0, ly=32.0, eta=0.4, seed=3))
    try:
        for _ in range(200):
            A.aap_step(h, 1)
            o = A.aap_observe(h)
            A.aap_clear_results(h)
            A.aap_measure(h, 1)
            r = A.aap_get_results(h)
            assert (r.samples, r.p[0], r.q[0]) == (1, o.phi, o.q)
    finally:
        A.aap_destroy(h)


@pytest.mark.parametrize("threads", [0, 512])
def test_measured_moments_are_the_sums_of_the_trace(threads):
    """The moments of p over a window from p(t) itself, bit for bit: powers by
    repeated rounded products, the fourth's last product added unrounded."""
    from fractions import Fraction

    kw = dict(n=1000, lx=32.0, ly=32.0, eta=0.4, seed=3, threads=threads)
    h1, h2 = A.aap_create(params(**kw)), A.aap_create(params(**kw))
    try:
        steps = 60
        A.aap_measure(h1, steps)
        sums = [0.0] * 4
        for p in A.aap_phi_trace(h2, steps)[:steps].tolist():
            sums[0] += p
            sums[1] += p * p
            sums[2] += p * p * p
            sums[3] = float(Fraction(p * p * p) * Fraction(p) + Fraction(sums[3]))
        r = A.aap_get_results(h1)
        assert r.samples == steps and list(r.p) == [s / steps for s in sums]
    finally:
        A.aap_destroy(h1)
        A.aap_destroy(h2)


def test_withheld_arrival_is_the_many_steps_kernels():
    h = A.aap_create(params(n=3000, lx=40.0, ly=40.0, eta=0.3, seed=23))
    try:
        A.aap_test_pipe_wait(20_000_000, 1)
        A.aap_step(h, 20)
        with pytest.raises(A.AapError) as e:
            A.aap_sync(h)
        assert e.value.code == A.AAP_ETIMEOUT
        assert list(A.aap_test_paths(h)[:2]) == [1, 20]
    finally:
        A.aap_test_pipe_wait(0, 0)
        A.aap_destroy(h)


@pytest.mark.parametrize("kw,w,front", [
    (dict(n=60000, lx=170.0, ly=160.0, eta=0.3, seed=31), 9.0, True),
    (dict(n=60000, lx=170.0, ly=160.0, eta=0.2, seed=32, model=A.AAP_NVM, by=1), 3.0, True),
    (dict(n=50000, lx=400.0, ly=380.0, eta=0.4, v=1.0, seed=33, model=A.AAP_LANGEVIN, bx=1, by=1), 14.0, True),
    (dict(n=9000, lx=60.0, ly=60.0, eta=0.3, seed=34, tile_w=64, tile_h=6), 20.0, False)])
def test_dense_tiles_are_split_and_lead(kw, w, front):
    """The states of the split-tile test: jobs beyond the tiles, and (where a
    tile has more own particles than two buffers hold) leading ones."""
    n, lx, ly = kw["n"], kw["lx"], kw["ly"]
    c = clustered_state(n // 4, lx, ly, 5, 0.3 * lx, 0.6 * ly, w)
    d = clustered_state(n // 8, lx, ly, 6, 0.9 * lx, 0.1 * ly, 2.0 * w)
    u = uniform_state(n - n // 4 - n // 8, lx, ly, 7)
    x, y, th = (np.concatenate(v) for v in zip(c, d, u))
    h = A.aap_create(params(threads=1024, **kw))
    try:
        A.aap_set_state(h, np.clip(x, 0.0, lx), np.clip(y, 0.0, ly), th.astype(np.float32), 0)
        lay = A.aap_get_layout(h)
        lead, jobs = A.aap_test_paths(h)[2:]
        assert jobs > lay.ntx * lay.nty and (lead > 0) == front
    finally:
        A.aap_destroy(h)


@pytest.mark.parametrize("side,dense,listed", [(330.0, True, True), (420.0, True, False), (330.0, False, False)])
def test_job_list_for_dense_states_of_few_tiles_per_sm(side, dense, listed):
    """Up to 12 tiles per SM (some 1,700 tiles of 8 x 8 cells) a state with a
    dense spot claims from the job list, beyond (2,700) and without one in
    raster order."""
    n = 120000
    h = A.aap_create(params(n=n, lx=side, ly=side, eta=0.3, seed=41, tile_w=8, tile_h=8, threads=1024))
    try:
        assert A.aap_test_paths(h)[3] == 0                  # the uniform start
        if dense:
            c = clustered_state(n // 4, side, side, 5, 0.3 * side, 0.6 * side, 6.0)
            u = uniform_state(n - n // 4, side, side, 7)
            x, y, th = (np.concatenate(v) for v in zip(c, u))
            A.aap_set_state(h, x, y, th.astype(np.float32), 0)
        assert (A.aap_test_paths(h)[3] > 0) == listed
    finally:
        A.aap_destroy(h)


def test_the_variant_follows_the_state_within_a_call():
    """A spot that spreads (straight paths) leaves the job list, and a ring
    that closes in takes it up: the state is looked at every 32 steps, through
    both variants' graphs, and the states equal the whole-block kernel's."""
    n, m, side = 1000000, 2500, 700.0
    g = np.random.default_rng(5)
    a = g.permutation(m) * (2.0 * np.pi / m) - np.pi
    u = uniform_state(n - m, side, side, 7)
    for first, radius, out in ((True, 2.0, 1.0), (False, 100.0, -1.0)):
        x, y = (np.concatenate([335.3 + radius * f(a), v]) for f, v in ((np.cos, u[0]), (np.sin, u[1])))
        th = np.concatenate([a if out > 0 else np.mod(a + 2.0 * np.pi, 2.0 * np.pi) - np.pi, u[2]]).astype(np.float32)
        states = []
        for threads in (1024, 512):
            h = A.aap_create(params(n=n, lx=side, ly=side, model=A.AAP_LANGEVIN, v=1.0, dt=1.0, eta=0.0, gamma=0.0, seed=6,
                                    tile_w=32, tile_h=16, threads=threads))
            try:
                A.aap_set_state(h, x, y, th, 0)
                if threads == 1024:
                    assert (A.aap_test_paths(h)[3] > 0) == first
                for _ in range(3):
                    A.aap_step(h, 32)
                A.aap_sync(h)
                A.aap_step(h, 0)
                if threads == 1024:
                    assert (A.aap_test_paths(h)[3] > 0) != first
                states.append(A.aap_get_state(h, n))
            finally:
                A.aap_destroy(h)
        for p, q in zip(*states):
            assert np.array_equal(p, q)


@pytest.mark.parametrize("batch,h,w,fused", [(1, 16, 16, True), (2, 128, 128, True), (4, 128, 128, True), (5, 128, 128, False)])
def test_small_predictions_are_fused(batch, h, w, fused):
    f = torch.full((batch, 3, h, w), 1.5, device="cuda")
    eta = torch.full((batch,), 0.4, device="cuda")
    s = A.aap_sur_create(A.aap_sur_params_default(nbx=w, nby=h, max_batch=batch))
    try:
        for _ in range(2):
            A.aap_sur_predict(s, f.data_ptr(), eta.data_ptr(), batch, 3, f.data_ptr())
        assert list(A.aap_sur_test_paths(s)) == ([6, 0] if fused else [0, 6])
    finally:
        A.aap_sur_destroy(s)


@pytest.mark.parametrize("sizes", [[(900, 1.0)] * 400, [(30000, 8.0), (30000, 0.5), (20000, 1.0), (300, 2.0), (60000, 4.0)]])
def test_ensemble_of_changing_systems_and_split_tiles(sizes):
    """The sort warps change the system of an output buffer with nearly every
    tile (400 replicas of a tile or two each, measured and not), and dense
    replicas beside dilute ones split their tiles: equal to the whole-block
    kernel's ensemble bit for bit."""
    out = []
    for threads in (1024, 512):
        ps = [params(n=n, lx=(n / rho) ** 0.5, ly=(n / rho) ** 0.5, eta=0.2 + 0.001 * r, seed=50 + r, threads=threads)
              for r, (n, rho) in enumerate(sizes)]
        e = A.aap_ens_create(ps)
        try:
            lays = [A.aap_ens_get_layout(e, r) for r in range(len(ps))]
            jobs = A.aap_ens_test_paths(e)[3]
            tiles = sum(v.ntx * v.nty for v in lays)
            if threads == 1024:
                assert jobs == 0 if len(ps) > 100 else jobs > tiles
            for steps in (1, 40):
                A.aap_ens_step(e, steps)
                A.aap_ens_measure(e, steps)
            res = [A.aap_ens_results(e, r) for r in range(len(ps))]
            out.append([v for r, p in enumerate(ps) for v in A.aap_ens_get_state(e, r, p.n)] +
                       [np.array(list(v.p) + list(v.q) + list(v.nbar)) for v in res] + [A.aap_ens_phi_mean(e)])
        finally:
            A.aap_ens_destroy(e)
    for a, b in zip(*out):
        assert np.array_equal(a, b)
