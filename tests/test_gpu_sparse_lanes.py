"""The edge-list step over its lane layouts: every stored label count, lists
shared by one to 32 lane groups, empty lists and a hub, variables that do not
fill a warp; and its deferred free energy with the stopping rule."""
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
    return binding, oracle


def graph(N, deg, L, sym, hub=0):
    d = synth.random_graph(N, N * deg, L, seed=N + 10 * deg + L, symmetric=sym, coupling_scale=1.0 / max(deg, 1))
    if hub:   # variable 0 joined to many, the last one to none
        rng = np.random.default_rng(N)
        keep = (d["src"] != N - 1) & (d["dst"] != N - 1)
        extra = 1 + rng.integers(0, N - 2, hub).astype(np.int32)
        d["src"] = np.concatenate([d["src"][keep], np.zeros(hub, np.int32)])
        d["dst"] = np.concatenate([d["dst"][keep], extra])
        d["w"] = np.concatenate([d["w"][keep], rng.uniform(0.0, 0.02, hub).astype(np.float32)])
    return d


def model(oracle, d):
    return oracle.Model.sparse(d["U"].astype(np.float64), d["mu"].astype(np.float64), d["src"].astype(np.int64),
                               d["dst"].astype(np.int64), d["w"].astype(np.float64))


def handle(binding, d, batch=1):
    crf = binding.CRF(binding.CRF_SPARSE, d["L"], 1, d["N"], batch=batch)
    crf.set_unary(np.tile(d["U"], (batch, 1)))
    crf.set_graph(d["mu"], d["src"], d["dst"], d["w"])
    return crf


@pytest.mark.parametrize("L", [1, 2, 3, 5, 8, 9, 13, 16, 18, 21, 24, 27, 32])
@pytest.mark.parametrize("N,deg,sym,hub", [(203, 3, True, 150), (77, 20, False, 60), (1, 0, True, 0),
                                           (9, 70, True, 0)])
def test_steps_and_trace(env, L, N, deg, sym, hub):
    binding, oracle = env
    d = graph(N, deg, L, sym, hub)
    m = model(oracle, d)
    eta, iters = 0.2, 4
    s_ref, F_ref = m.parallel_prox(eta, iters)
    with handle(binding, d) as crf:
        crf.iterate(iters, eta=eta, reset=True)
        q = crf.marginals()[0].astype(np.float64)
        trace, F = crf.free_energy_trace(iters)[0], crf.free_energy()[0]
    assert np.abs(q - np.exp(s_ref)).max() <= 1e-5
    assert H.f_close(trace, F_ref[:-1], N, 1e-6)
    assert H.f_close(F, F_ref[-1], N, 1e-6)


@pytest.mark.parametrize("N,L", [(20011, 2), (30011, 21)])
def test_more_variables_than_one_round_of_blocks(env, N, L):
    """Blocks take several rounds (the last one partly filled)."""
    binding, oracle = env
    d = graph(N, 4, L, True)
    s_ref, F_ref = model(oracle, d).parallel_prox(0.1, 2)
    with handle(binding, d) as crf:
        crf.iterate(2, eta=0.1, reset=True)
        q = crf.marginals()[0].astype(np.float64)
        trace = crf.free_energy_trace(2)[0]
    assert np.abs(q - np.exp(s_ref)).max() <= 1e-5
    assert H.f_close(trace, F_ref[:-1], N, 1e-6)


def test_stopping_rule(env):
    binding, oracle = env
    d = graph(500, 4, 6, True)
    eta, tol, iters = 0.15, 2e-3, 60
    m = model(oracle, d)
    F = m.parallel_prox(eta, iters)[1]
    stop = next((t + 1 for t in range(1, iters) if abs(F[t] - F[t - 1]) <= tol * abs(F[t])), iters)
    with handle(binding, d, batch=2) as crf:
        took = crf.iterate(iters, eta=eta, reset=True, rel_tol=tol, want_iters=True)
        q = crf.marginals().astype(np.float64)
    assert list(took) == [stop, stop]
    for b in range(2):
        assert np.abs(q[b] - np.exp(m.parallel_prox(eta, stop)[0])).max() <= 1e-5


def test_new_graph_on_a_handle_that_replays(env):
    """A recorded step loop is not replayed on the arrays of an earlier graph."""
    binding, oracle = env
    a, b = graph(300, 3, 5, True), graph(300, 30, 5, False)
    b["U"] = a["U"]
    with handle(binding, a) as crf:
        crf.use_graphs(True)
        crf.iterate(5, eta=0.2, reset=True)
        crf.set_graph(b["mu"], b["src"], b["dst"], b["w"])
        crf.iterate(5, eta=0.2, reset=True)
        q = crf.marginals()[0].astype(np.float64)
    assert np.abs(q - np.exp(model(oracle, b).parallel_prox(0.2, 5)[0])).max() <= 1e-5
