"""The FP32 dense step where its tiles, chunks and k ranges end: rows around
128, k around 8, two stored labels on odd instances (their rows start off a
16-byte boundary), label counts of both lane layouts, clusters of one to eight
CTAs; and its deferred free energy with the stopping rule."""
import numpy as np
import pytest

from paper_1511_06103_gb300 import synth
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.init()
    from paper_1511_06103_gb300 import binding, build
    build.build()
    import oracle
    oracle.build()
    return binding, oracle, torch


def instance(h, w, L, seed, mu=None):
    rng = np.random.default_rng(seed)
    N = h * w
    yy, xx = np.meshgrid(np.arange(h), np.arange(w), indexing="ij")
    feats = np.concatenate([np.stack([xx, yy], -1).reshape(N, 2), rng.uniform(0, 60, (N, 3))], 1)
    m = (1.0 - np.eye(L)) + 0.5 * synth.symmetric_uniform(L, rng) if mu is None else mu
    return dict(N=N, L=L, U=synth.unary_from_logits(rng.normal(0, 2, (N, L))).astype(np.float32),
                mu=m.astype(np.float32), feats=feats.astype(np.float32), theta=(3.0, 13.0))


def model(oracle, d):
    K = oracle.dense_gauss_kernel(d["feats"].astype(np.float64), *d["theta"])
    return oracle.Model.dense(d["U"].astype(np.float64), d["mu"].astype(np.float64), K)


@pytest.mark.parametrize("h,w,L,B", [(1, 1, 3, 1), (1, 7, 2, 3), (1, 127, 5, 1), (2, 64, 16, 1), (3, 43, 20, 1),
                                     (17, 15, 2, 3), (16, 23, 12, 2), (5, 53, 24, 2), (41, 40, 21, 1),
                                     (49, 47, 4, 1)])
def test_steps_and_trace(env, h, w, L, B):
    binding, oracle, torch = env
    ds = [instance(h, w, L, 100 * h + 10 * w + L)]
    ds += [instance(h, w, L, 7 + b, ds[0]["mu"]) for b in range(1, B)]
    iters, eta = 4, 0.2
    with binding.CRF(binding.CRF_DENSE_GAUSS, L, h, w, batch=B) as crf:
        crf.set_unary(np.stack([d["U"] for d in ds]))
        crf.set_pairwise(ds[0]["mu"], np.stack([d["feats"] for d in ds]), theta=np.array(ds[0]["theta"], np.float32))
        crf.iterate(1, eta=eta, reset=True)
        q1 = crf.marginals().astype(np.float64)
        crf.iterate(iters, eta=eta, reset=True)
        q = crf.marginals().astype(np.float64)
        trace, F = crf.free_energy_trace(iters), crf.free_energy()
    for b, d in enumerate(ds):
        m = model(oracle, d)
        s_ref, F_ref = m.parallel_prox(eta, iters)
        assert np.abs(q1[b] - np.exp(m.parallel_prox(eta, 1)[0])).max() <= 1e-6
        assert np.abs(q[b] - np.exp(s_ref)).max() <= 1e-5
        assert H.f_close(trace[b], F_ref[:-1], d["N"], 1e-6)
        assert H.f_close(F[b], F_ref[-1], d["N"], 1e-6)


def test_stopping_rule(env):
    """Instances of a batch stop at their own step, their state as it was then."""
    binding, oracle, torch = env
    ds = [instance(12, 25, 6, 3)]
    ds.append(instance(12, 25, 6, 4, ds[0]["mu"]))
    ds[1]["U"] = (0.2 * ds[1]["U"]).astype(np.float32)
    eta, tol, iters = 0.15, 2e-3, 60
    with binding.CRF(binding.CRF_DENSE_GAUSS, 6, 12, 25, batch=2) as crf:
        crf.set_unary(np.stack([d["U"] for d in ds]))
        crf.set_pairwise(ds[0]["mu"], np.stack([d["feats"] for d in ds]), theta=np.array(ds[0]["theta"], np.float32))
        took = crf.iterate(iters, eta=eta, reset=True, rel_tol=tol, want_iters=True)
        q = crf.marginals().astype(np.float64)
    for b, d in enumerate(ds):
        m = model(oracle, d)
        F = m.parallel_prox(eta, iters)[1]
        stop = next((t + 1 for t in range(1, iters) if abs(F[t] - F[t - 1]) <= tol * abs(F[t])), iters)
        assert took[b] == stop
        assert np.abs(q[b] - np.exp(m.parallel_prox(eta, stop)[0])).max() <= 1e-5
