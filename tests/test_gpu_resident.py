"""The one-launch loop of small grids where its slabs, pixels per thread and
blocks of steps end: fewer rows than CTAs, CTAs without rows, one column, slabs
at the limits of one and two pixels a thread, step counts around 32 and 64."""
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


def model(oracle, d):
    return oracle.Model.grid(d["U"].astype(np.float64), d["mu"].astype(np.float64), d["w"].astype(np.float64),
                             d["H"], d["W"], d["conn"])


def handle(binding, ds):
    d = ds[0]
    crf = binding.CRF(binding.CRF_GRID8 if d["conn"] == 8 else binding.CRF_GRID4, d["L"], d["H"], d["W"],
                      batch=len(ds))
    crf.set_unary(np.stack([x["U"] for x in ds]))
    crf.set_pairwise(d["mu"], np.stack([x["w"] for x in ds]))
    return crf


@pytest.mark.parametrize("Hh,Ww,L,conn,sym,iters", [
    (1, 40, 2, 4, True, 2), (2, 1, 3, 8, False, 5), (9, 33, 2, 8, True, 32), (13, 21, 1, 4, True, 33),
    (8, 512, 16, 8, True, 31), (32, 128, 16, 8, True, 35), (16, 256, 11, 4, False, 64), (16, 257, 7, 8, False, 65), (24, 341, 5, 8, True, 97),
    (8, 1024, 4, 8, False, 34), (24, 520, 4, 4, True, 40), (40, 800, 2, 8, False, 66), (17, 512, 13, 8, False, 36)])
def test_against_the_oracle(env, Hh, Ww, L, conn, sym, iters):
    binding, oracle = env
    d = synth.random_grid(Hh, Ww, L, conn, seed=31 * Hh + L, symmetric=sym, coupling_scale=0.3)
    s_ref, F_ref = model(oracle, d).parallel_prox(0.2, iters)
    with handle(binding, [d]) as crf:
        n0 = crf.launch_count()
        crf.iterate(iters, eta=0.2)
        resident = crf.launch_count() - n0 <= 2
        q = crf.marginals()[0].astype(np.float64)
        trace, F = crf.free_energy_trace(iters)[0], crf.free_energy()[0]
    # 17 x 512 x 13 has 1536 pixels a slab, past the limit of its label count;
    # 8 x 512 x 16 wants 2 x 3 x 514 cells of 80 bytes, past the shared memory
    assert resident == ((Hh, Ww, L) not in ((17, 512, 13), (8, 512, 16)))
    assert np.abs(q - np.exp(s_ref)).max() <= 1e-5
    assert H.f_close(trace, F_ref[:-1], Hh * Ww, 1e-6)
    assert H.f_close(F, F_ref[-1], Hh * Ww, 1e-6)


@pytest.mark.parametrize("Hh,Ww,L", [(11, 60, 2), (20, 130, 6)])
def test_stopping_rule_per_instance(env, Hh, Ww, L):
    binding, oracle = env
    ds = [synth.random_grid(Hh, Ww, L, 8, seed=5, coupling_scale=0.3),
          synth.random_grid(Hh, Ww, L, 8, seed=6, coupling_scale=0.3, unary_scale=0.3)]
    ds[1]["mu"] = ds[0]["mu"]
    eta, tol, iters = 0.15, 2e-3, 80
    with handle(binding, ds) as crf:
        took = crf.iterate(iters, eta=eta, reset=True, rel_tol=tol, want_iters=True)
        q = crf.marginals().astype(np.float64)
        trace = crf.free_energy_trace(iters)
    for b, d in enumerate(ds):
        m = model(oracle, d)
        F = m.parallel_prox(eta, iters)[1]
        stop = next((t + 1 for t in range(1, iters) if abs(F[t] - F[t - 1]) <= tol * abs(F[t])), iters)
        assert took[b] == stop
        assert np.abs(q[b] - np.exp(m.parallel_prox(eta, stop)[0])).max() <= 1e-5
        assert H.f_close(trace[b, :stop], F[:stop], Hh * Ww, 1e-6)
