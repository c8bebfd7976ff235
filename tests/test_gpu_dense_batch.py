"""Batches of fully connected models, FP32: an instance has the same bits alone and
in a batch, whatever number of CTAs takes its tiles' shares of k; each stops at its
own step; and a batch whose row tiles fit the chip takes about as long as one CTA
takes for a tile."""
import numpy as np
import pytest

from paper_1511_06103_gb300 import synth

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


def instances(B, h, w, L, seed):
    rng = np.random.default_rng(seed)
    yy, xx = np.meshgrid(np.arange(h), np.arange(w), indexing="ij")
    pos = np.broadcast_to(np.stack([xx, yy], -1).reshape(1, h * w, 2), (B, h * w, 2))
    feats = np.concatenate([pos, rng.uniform(0, 60, (B, h * w, 3))], -1).astype(np.float32)
    U = synth.unary_from_logits(rng.normal(0, 2, (B, h * w, L))).astype(np.float32)
    mu = ((1.0 - np.eye(L)) + 0.5 * synth.symmetric_uniform(L, rng)).astype(np.float32)
    return U, mu, feats


def solve(binding, U, mu, feats, h, w, bf16=False, **kw):
    B, _, L = U.shape
    with binding.CRF(binding.CRF_DENSE_GAUSS, L, h, w, batch=B,
                     precision=binding.CRF_BF16 if bf16 else binding.CRF_FP32) as crf:
        crf.set_unary(U)
        crf.set_pairwise(mu, feats, theta=np.array([3.0, 13.0], np.float32))
        n = kw.pop("iters")
        took = crf.iterate(n, eta=0.2, reset=True, refine_fp32=2 if bf16 else 0, want_iters=True, **kw)
        return crf.log_marginals(), crf.free_energy_trace(n), crf.free_energy(), took


@pytest.mark.parametrize("B,h,w,L,bf16", [(40, 8, 8, 5, False), (130, 9, 9, 2, False), (24, 11, 11, 21, False),
                                          (64, 11, 11, 3, False), (20, 16, 16, 21, False), (33, 16, 17, 12, False),
                                          (64, 16, 16, 20, False), (16, 22, 23, 24, False), (30, 30, 30, 8, False),
                                          (9, 30, 31, 16, False), (5, 41, 40, 21, False), (5, 48, 47, 4, False),
                                          (64, 16, 16, 18, True), (200, 1, 7, 3, False)])
def test_alone_and_in_a_batch(env, B, h, w, L, bf16):
    binding, oracle, torch = env
    U, mu, feats = instances(B, h, w, L, B + L)
    s, tr, F, _ = solve(binding, U, mu, feats, h, w, bf16, iters=4)
    for b in (0, B // 2, B - 1):
        s1, tr1, F1, _ = solve(binding, U[b:b + 1], mu, feats[b:b + 1], h, w, bf16, iters=4)
        assert np.array_equal(s[b], s1[0]) and np.array_equal(tr[b], tr1[0]) and F[b] == F1[0]
    if not bf16:
        K = oracle.dense_gauss_kernel(feats[B - 1].astype(np.float64), 3.0, 13.0)
        m = oracle.Model.dense(U[B - 1].astype(np.float64), mu.astype(np.float64), K)
        ref = np.exp(m.parallel_prox(float(np.float32(0.2)), 4)[0])
        assert np.abs(np.exp(s[B - 1].astype(np.float64)) - ref).max() <= 1e-5


@pytest.mark.parametrize("B,h,w,L", [(40, 8, 9, 6), (24, 16, 16, 21)])
def test_stopping_rule(env, B, h, w, L):
    binding, oracle, torch = env
    U, mu, feats = instances(B, h, w, L, 3)
    U *= np.linspace(0.1, 1.0, B, dtype=np.float32)[:, None, None]
    s, _, _, took = solve(binding, U, mu, feats, h, w, iters=60, rel_tol=1e-4)
    assert len(set(took.tolist())) > 1
    for b in (0, B // 3, B - 1):
        s1, _, _, t1 = solve(binding, U[b:b + 1], mu, feats[b:b + 1], h, w, iters=60, rel_tol=1e-4)
        assert took[b] == t1[0] and np.array_equal(s[b], s1[0])


def test_time_of_a_batch(env):
    """64 instances of N = 256 are 128 row tiles, a CTA each: eight times the k of one
    CTA of a lone instance's cluster, beside a fixed part worth 460 k in both and three
    rounds worth 100, so (256 + 460 + 300) / (32 + 460) = 2.1 times its time; 5 allowed."""
    binding, oracle, torch = env
    ms = {}
    for B in (1, 64):
        U, mu, feats = instances(B, 16, 16, 21, 5)
        with binding.CRF(binding.CRF_DENSE_GAUSS, 21, 16, 16, batch=B) as crf:
            crf.set_unary(U)
            crf.set_pairwise(mu, feats, theta=np.array([3.0, 13.0], np.float32))
            crf.profile()
            ms[B] = np.inf
            for _ in range(8):
                crf.iterate(40, eta=0.2, reset=True)
                ms[B] = min(ms[B], crf.profile_read()[0])
    assert ms[64] <= 5 * ms[1], ms
