"""Row conversions and the initial state at the edges of their blocks: one row
to a few rows past a block for every stored label count, buffers that start off
a 16-byte boundary, page-locked buffers used in place."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.init()
    from paper_1511_06103_gb300 import binding, build
    build.build()
    return binding, torch


def softmax(U):
    z = np.exp(-(U - U.min(-1, keepdims=True)).astype(np.float64))
    return z / z.sum(-1, keepdims=True)


@pytest.mark.parametrize("L", [1, 2, 3, 4, 6, 8, 11, 16, 19, 21, 24, 26, 31, 32])
@pytest.mark.parametrize("H,W", [(1, 1), (3, 43), (1, 127), (8, 32), (27, 19), (1, 1025)])
@pytest.mark.parametrize("where", ["device", "device_odd", "pinned_odd", "pageable"])
def test_unaries_in_marginals_out(env, L, H, W, where):
    binding, torch = env
    N = H * W
    U = np.random.default_rng(N + L).normal(0, 3, (N, L)).astype(np.float32)
    n = N * L

    def buffer(src=None):
        off = 1 if where.endswith("odd") else 0
        t = torch.empty(n + off, device="cuda" if where.startswith("device") else "cpu")
        if where.startswith("pinned"):
            t = t.pin_memory()
        v = t[off:].view(1, N, L)
        if src is not None:
            v.copy_(torch.from_numpy(src).view(1, N, L))
        return v

    with binding.CRF(binding.CRF_GRID4, L, H, W) as crf:
        crf.set_unary(buffer(U))
        q, s = buffer(), buffer()
        crf.marginals(q)
        crf.log_marginals(s)
        torch.cuda.synchronize()
        ref = softmax(U)
        # FP32 log-sum-exp of L terms and the exponential of the result
        assert np.abs(q.cpu().numpy()[0] - ref).max() <= 4e-6
        assert np.abs(s.cpu().numpy()[0] - np.log(ref)).max() <= 2e-6 * np.abs(np.log(ref)).max() + 2e-6
        crf.set_state(s)   # rows in and out unchanged
        t = buffer()
        crf.log_marginals(t)
        torch.cuda.synchronize()
        assert torch.equal(t, s)


@pytest.mark.parametrize("conn", [4, 8])
@pytest.mark.parametrize("H,W,B", [(1, 1, 1), (1, 300, 2), (300, 1, 2), (17, 31, 3)])
def test_weights_of_edges_that_leave_the_image_are_ignored(env, conn, H, W, B):
    """F of uniform marginals is linear in the weights of existing edges."""
    binding, torch = env
    nd = conn // 2
    w = np.random.default_rng(H + W).uniform(0.5, 1.5, (B, nd, H, W)).astype(np.float32)
    dy, dx = (0, 1, 1, 1), (1, 0, 1, -1)
    tot = np.zeros(B)
    for k in range(nd):
        y, x = np.meshgrid(np.arange(H), np.arange(W), indexing="ij")
        ok = (y + dy[k] < H) & (x + dx[k] >= 0) & (x + dx[k] < W)
        tot += (w[:, k].astype(np.float64) * ok).sum((1, 2))
    mu = np.array([[0, 1, 2], [1, 0, 1], [2, 1, 0]], np.float32)
    with binding.CRF(binding.CRF_GRID8 if conn == 8 else binding.CRF_GRID4, 3, H, W, batch=B) as crf:
        crf.set_unary(np.zeros((B, H * W, 3), np.float32))
        crf.set_pairwise(mu, w)
        F = crf.free_energy()
    assert np.allclose(F, tot * mu.mean() - H * W * np.log(3.0), rtol=2e-6, atol=2e-6 * H * W)
