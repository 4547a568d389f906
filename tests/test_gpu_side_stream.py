"""Handles made on a stream of their own (not ordered with the default stream)
while the default stream is busy: everything their creation uploads or clears
goes through their own stream, so they give the same results bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

import paper_2211_15630_gb300 as A
from tests.gpu_helpers import params

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def lib():
    return A.load()


def system(stream):
    n = 3000
    h = A.aap_create(params(n=n, lx=40.0, ly=37.0, eta=0.3, seed=4), stream)
    A.aap_step(h, 40)
    out = A.aap_get_state(h, n)
    A.aap_destroy(h)
    return list(out)


def ensemble(stream):
    ps = [params(n=n, lx=(n / rho) ** 0.5, ly=(n / rho) ** 0.5, eta=0.2, seed=5 + r)
          for r, (n, rho) in enumerate([(9000, 8.0), (9000, 0.5), (300, 2.0), (20000, 4.0)])]
    e = A.aap_ens_create(ps, stream)
    A.aap_ens_measure(e, 40)
    out = [v for r, p in enumerate(ps) for v in A.aap_ens_get_state(e, r, p.n)] + [A.aap_ens_phi_mean(e)]
    A.aap_ens_destroy(e)
    return out


def surrogate(stream):
    g = np.random.default_rng(6)
    s = A.aap_sur_create(A.aap_sur_params_default(nbx=32, nby=48, max_batch=2, conserve=3), stream)
    with torch.cuda.stream(torch.cuda.ExternalStream(stream) if stream else torch.cuda.default_stream()):
        f = torch.tensor(g.uniform(1.0, 2.0, (2, 3, 48, 32)), dtype=torch.float32).pin_memory().cuda(non_blocking=True)
        t = f * 1.1
        eta = torch.full((2,), 0.4, device="cuda")
    loss = A.aap_sur_train_step(s, f.data_ptr(), t.data_ptr(), eta.data_ptr(), 2)
    out = [np.array(loss), A.aap_sur_get_grads(s), A.aap_sur_get_params(s)]
    A.aap_sur_destroy(s)
    return out


@pytest.mark.parametrize("work", [system, ensemble, surrogate])
def test_same_results_beside_a_busy_default_stream(work):
    expect = work(None)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    torch.cuda._sleep(400_000_000)          # some 0.2 s on the default stream
    got = work(side.cuda_stream)
    torch.cuda.synchronize()
    assert len(got) == len(expect)
    for a, b in zip(expect, got):
        assert np.array_equal(a, b)
