"""Forbidden labels (infinite unary costs) in the server: log q = -inf stays
log q = -inf, and the other labels' marginals are those of the model, in every
group of requests."""
import numpy as np
import pytest

from paper_1511_06103_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def oracle():
    import oracle
    oracle.build()
    return oracle


@pytest.mark.parametrize("L,conn,sym", [(2, 4, True), (3, 4, True), (8, 8, True), (13, 8, True), (21, 8, True),
                                        (8, 8, False), (24, 8, True)])
def test_forbidden_labels(oracle, L, conn, sym):
    from paper_1511_06103_gb300 import binding
    H, W, eta = 19, 37, 0.2
    d = synth.random_grid(H, W, L, conn, seed=40 + L, symmetric=sym)
    rng = np.random.default_rng(L)
    U = d["U"].reshape(H * W, L).astype(np.float32)
    ban = rng.random((H * W, L)) < 0.3
    ban[np.arange(H * W), rng.integers(0, L, H * W)] = False   # one label is left everywhere
    U[ban] = np.inf
    with binding.Server(1 << 26) as srv:
        t = srv.submit(U, d["mu"], d["w"], H, W, conn, eta=eta, max_iters=1)
        for _ in range(100):
            srv.step(1)
            srv.sync()
            if srv.poll(t)[0] == 2:
                break
        st, F, it, q = srv.poll(t)
    assert st == 2 and it == 1
    # a cost of 1e4 leaves e^-10000 of a label: 0 in FP32 and FP64
    m = oracle.Model.grid(np.where(ban, 1e4, U).astype(np.float64), d["mu"].astype(np.float64),
                          d["w"].astype(np.float64), H, W, conn)
    ref = np.exp(m.parallel_prox(float(np.float32(eta)), 1)[0]).reshape(H * W, L)
    assert np.all(q[ban] == 0.0)
    assert np.abs(q - ref).max() <= 1e-5
